// Device-side helpers shared by the fehmm kernels: vector traits, warp/block reductions
// and the compressible neo-Hookean law of the paper's Sec. 6 in the factored form used by
// the kernels.
//
// Neo-Hookean law (Eq. NH-free-energy and the closed forms for S and CC that follow it):
//   psi = lam/4 (J^2 - 1) - (lam/2 + mu) ln J + mu/2 (tr C - 3)
//   S   = lam/2 (J^2 - 1) C^-1 + mu (I - C^-1)
// With F C^-1 = F^-T (written Fit) and F C^-1 F^T = I these give, exactly,
//   P = F S = mu F + hb Fit,                       hb = lam (J^2 - 1)/2 - mu
//   A_iJkL = dP_iJ/dF_kL = mu d_ik d_JL - hb Fit_iL Fit_kJ + gm Fit_iJ Fit_kL,  gm = lam J^2
// which is delta_ik S_JL + F_iI F_kK CC_IJKL with CC = [lam (J^2-1) - 2 mu] dC^-1/dC
// + lam J^2 C^-1 (x) C^-1 (Eq. Aijkl-NeoHook) after contracting with F.  2D is plane strain
// (F_33 = 1): the same formulas hold for the in-plane 2x2 blocks.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fehmm {

constexpr int kMaxPhase = 4;
constexpr int kStatusOk = 0, kStatusNewtonCap = 1, kStatusJNonPos = 2, kStatusPcgBreakdown = 3,
              kStatusNonFinite = 4, kStatusPcgCap = 5,
              kStatusNegCurv = 6,  // internal: truncated Newton-correction PCG
              kStatusBadPhase = 7;  // a device-supplied phase id >= kMaxPhase (nothing solved)
constexpr int kFlagNoTangent = 1, kFlagFromCommitted = 2, kFlagEnergy = 4;
// Newton globalisation: after an update that makes det F <= 0 somewhere (or the residual
// non-finite) the step is halved, up to this many times, before the RVE is reported failed.
constexpr int kMaxStepHalvings = 8;
// Newton cap of each load-continuation stage of a retried solve (at least max_newton): a retry
// recovers a usable state even when max_newton = 1 (the alternating scheme).
constexpr int kRetryNewtonCap = 25;

template <typename T> struct vec2_of;
template <> struct vec2_of<float> { using type = float2; };
template <> struct vec2_of<double> { using type = double2; };
template <typename T> using vec2_t = typename vec2_of<T>::type;

template <typename T>
__device__ __forceinline__ vec2_t<T> mk2(T x, T y) {
  vec2_t<T> v;
  v.x = x;
  v.y = y;
  return v;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// FP64 sums of NV values over a block of up to 16 warps; every thread receives the totals.  An FP64 warp instruction
// holds its sub-partition for 64 cycles, so each sum is formed once: the values are dealt to the lanes in the first
// levels of the shuffle tree (16 additions for ten values, where a tree for each takes 50), and the warps add up
// different values of the block.  buf: kBlockSumDoubles doubles of shared memory; consecutive calls may use the same
// (each barrier orders one part's reads before the next call's writes).  Two barriers.
constexpr int kBlockSumDoubles = 170;
template <int NV>
__device__ __forceinline__ void block_sum_fp64(double (&v)[NV], double* buf) {
  constexpr int P = NV <= 1 ? 1 : NV <= 8 ? 8 : 16, kShift = NV <= 1 ? 5 : NV <= 8 ? 2 : 1;
  static_assert(NV <= 10, "the buffer holds ten values");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double a[P];
#pragma unroll
  for (int k = 0; k < P; ++k) a[k] = k < NV ? v[k] : 0.0;
  int o = 16;
#pragma unroll
  for (int cnt = P / 2; cnt >= 1; cnt /= 2) {
    const bool upper = lane & o;
#pragma unroll
    for (int j = 0; j < cnt; ++j) {
      const double send = upper ? a[j] : a[j + cnt], keep = upper ? a[j + cnt] : a[j];
      a[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    o >>= 1;
  }
#pragma unroll
  for (int q = 16 / P; q >= 1; q >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], q);
  const int held = lane >> kShift;  // the value this lane holds
  if ((lane & ((1 << kShift) - 1)) == 0 && held < NV) buf[16 * held + warp] = a[0];
  __syncthreads();
  for (int k = warp; k < NV; k += nw) {
    double t = lane < nw ? buf[16 * k + lane] : 0.0;
    for (int q = 8; q >= 1; q >>= 1)
      if (q < nw) t += __shfl_xor_sync(0xffffffffu, t, q);
    if (lane == 0) buf[160 + k] = t;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = buf[160 + k];
}

__device__ __forceinline__ bool positive_fp64(double x) {  // x > 0 (false for NaN) without an FP64 instruction
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}

// The two inner products of a PCG step over a block of up to 16 warps, and the tests on them.  Each thread's
// partial and the warp's shuffle tree are in T (FP32 in mixed mode); warp 0 adds the warp sums in FP64 (lanes 0-15 the
// first, lanes 16-31 the second product, in a fixed order) and compares them there, and the block receives them
// rounded to T with the outcome of the tests as flags.  (With the FP64 sums broadcast, every warp converted and
// compared them itself: five FP64-pipe instructions a warp, at 16 warps about 1300 cycles of an iteration.)
// stop is compared with the first sum and needed by warp 0 only, as wide, the unrounded first sum, is valid there.
// buf: kDotDoubles doubles; consecutive calls may use the same.  Two barriers.
constexpr int kDotDoubles = 36;
constexpr int kDotNonNeg = 1, kDotPos = 2, kDotFinite = 4, kDotStop = 8, kDotCurvPos = 16;
template <typename T>
__device__ __forceinline__ int block_dot2(T a, T b, double* buf, double stop, T& sa, T& sb, double& wide) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* part = reinterpret_cast<T*>(buf);
  T* out = reinterpret_cast<T*>(buf + 32);
  int* flags = reinterpret_cast<int*>(buf + 34);
  a = warp_sum(a);
  b = warp_sum(b);
  if (lane == 0) {
    part[warp] = a;
    part[16 + warp] = b;
  }
  __syncthreads();
  wide = 0.0;
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    double v = (lane & 15) < nw ? (double)part[lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
      if (o < nw) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) == 0) out[lane >> 4] = (T)v;
    wide = __shfl_sync(0xffffffffu, v, 0);
    const double curv = __shfl_sync(0xffffffffu, v, 16);
    if (lane == 0) {
      const long long g = __double_as_longlong(wide);  // ordered as the doubles where both are >= 0
      const bool zero = (g << 1) == 0, pos = positive_fp64(wide);
      *flags = (pos || zero ? kDotNonNeg : 0) | (pos ? kDotPos : 0) |
               ((g & 0x7ff0000000000000ll) != 0x7ff0000000000000ll ? kDotFinite : 0) |
               ((pos || zero) && g <= __double_as_longlong(stop) ? kDotStop : 0) | (positive_fp64(curv) ? kDotCurvPos : 0);
    }
  }
  __syncthreads();
  sa = out[0];
  sb = out[1];
  return *flags;
}

// FP64 reciprocals without the FP64 instructions of a division (about nine; an FP64 instruction holds an SM
// sub-partition for 64 cycles): the hardware's FP32 approximation x0 (rcp.approx, error at most one FP32 ulp), then one
// step of the hyperpower iteration of order 3, x = x0 + x0 (e + e^2) with e = 1 - a x0.  Its error is e^3, below 2^-65
// of the result, so what is left is the rounding of the last operation: within one ulp of 1 / a.

// 1 / x for every x: normal positive x below 2^1018 with its exponent split off, which keeps the mantissa in FP32's
// range; any other (zero, subnormal, negative, infinite, NaN) by the division.
__device__ __forceinline__ double recip_d(double x) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (e == 0 || e > 2040 || hi < 0) return 1.0 / x;
  const double m = __hiloint2double((hi & 0xfffff) | (1023 << 20), __double2loint(x));
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((float)m));
  double q = (double)f;
  const double err = fma(-m, q, 1.0);
  q = fma(q, fma(err, err, err), q);
  return __hiloint2double(__double2hiint(q) + ((1023 - e) << 20), __double2loint(q));
}

// a / x by recip_d.  A subnormal x, whose reciprocal may overflow where the quotient does not (a CG that started from
// sums of 1e-300), takes the division, as do the others that recip_d divides for.
__device__ __forceinline__ double div_d(double a, double x) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (e == 0 || e > 2040 || hi < 0) return a / x;
  return a * recip_d(x);
}

// 1/J for the FP64 stress of the residuals, J in FP32's normal range: 2^-126 <= J < 2^126.  Conversions are FP64-pipe
// instructions too, so J's FP32 value and the reciprocal's FP64 value are put together from their bits there: three
// FP64 instructions in all.  Negative J of that range by conversions, as accurate.  A smaller |J| (a collapsed element)
// gives a non-finite result, which the Newton loop treats like J <= 0, a larger one zero.
__device__ __forceinline__ double recip_fp64(double J) {
  float r;
  double x;
  const int hi = __double2hiint(J);
  if ((unsigned)(hi - (897 << 20)) < (252u << 20)) {
    const float f = __uint_as_float(__funnelshift_l(__double2loint(J), hi, 3) + 0x40000000u);  // exponent bias 1023 -> 127
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
    const unsigned b = __float_as_uint(r);
    x = __hiloint2double((int)(b >> 3) + (896 << 20), (int)(b << 29));
  } else {
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"((float)J));
    x = (double)r;
  }
  const double e = fma(-J, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

// 1/J at the tangent's precision: FP32 through the hardware approximate reciprocal (about one
// FP32 ulp, ample for an FP32 tangent), FP64 as a plain division.
template <typename T>
__device__ __forceinline__ T recip_T(T J) {
  if constexpr (sizeof(T) == 4) {
    return __fdividef(1.f, J);
  } else {
    return 1.0 / J;
  }
}

// Lame constants from (E, nu), as in the paper's material table (Sec. 6).
__host__ __device__ inline void lame_from_E_nu(double E, double nu, double& lam, double& mu) {
  lam = E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu));
  mu = E / (2.0 * (1.0 + nu));
}

// 2D plane-strain point quantities: J, Fit = F^-T, hb, gm (see header comment).
template <typename T>
struct NH2 {
  T J, f00, f01, f10, f11;  // Fit
  T hb, gm;
};

template <typename T>
__device__ __forceinline__ NH2<T> nh2_eval(T F00, T F01, T F10, T F11, T lam, T mu) {
  NH2<T> r;
  r.J = F00 * F11 - F01 * F10;
  const T iJ = recip_T(r.J);
  r.f00 = F11 * iJ;
  r.f01 = -F10 * iJ;
  r.f10 = -F01 * iJ;
  r.f11 = F00 * iJ;
  const T J2 = r.J * r.J;
  r.hb = T(0.5) * lam * (J2 - T(1)) - mu;
  r.gm = lam * J2;
  return r;
}

}  // namespace fehmm
