"""The work that a user of this framework has it do, as a list of measurable cases.

Kinds of case and what each stands for in real use:

  rve2d     one batched 2D RVE solve (stress, tangent, fluctuations) of a macro iteration: the first
            one of a load step, started from the committed state of the step before
  noalloc   the same for callers that cannot allocate: fehmm_rve2d_solve_fp64_noalloc
  rve3d     one batched 3D RVE solve of a macro iteration
  training  stress and energy of 3D RVEs at sampled stretches by load continuation from zero, which
            is how the surrogate's training data are made
  macro     the macro part of an iteration: Fbar at the quadrature points, residual and tangent
            assembly, the CG solve of the Newton correction
  mlp       one training step of the surrogate network (loss, gradient, AdamW)
  surrogate stress, tangent and energy of the trained surrogate at many macro points
  step      one whole load step of the two-scale driver, from the previous step's state

Sizes are those of the workloads, tests and benchmark of this repository.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1908_08292_gb300 as fe
from paper_1908_08292_gb300 import surrogate as su
from paper_1908_08292_gb300.driver import LoadStepDriver

F64, F32, I32 = torch.float64, torch.float32, torch.int32


def listed():
    return [
        # one macro iteration of the smallest two-scale problem: 4 x 4 macro elements, one 8 x 8
        # microstructure at all 64 points, FP64: few points, latency counts
        dict(name="rve2d_64x8_fp64", kind="rve2d", n_qp=64, sizes="8", precision="fp64", law=0, bc=0, shared=True),
        # the headline: 32 x 32 macro elements, 4096 points, a 32 x 32 microstructure of its own at each
        dict(name="rve2d_4096x32_mixed", kind="rve2d", n_qp=4096, sizes="32", precision="mixed", law=0, bc=0,
             shared=False),
        # an uneven batch of a mesh study: odd number of points, grids with and without a multigrid hierarchy
        dict(name="rve2d_ragged_mixed", kind="rve2d", n_qp=333, sizes="6,10,12,16,20,24,30", precision="mixed", law=0,
             bc=0, shared=False),
        # a caller with a fixed footprint: 16 x 16 (the largest grid of that entry), FP64, block-Jacobi
        dict(name="noalloc_150x16_fp64", kind="noalloc", n_qp=150, sizes="16"),
        # a macro iteration of the uneven 3D batch: 4^3 macro elements, 512 points of 8^3, 12^3 and 16^3
        dict(name="rve3d_512_uneven_mixed", kind="rve3d", n_qp=512, sizes="8,12,16", precision="mixed", law=0, bc=0),
        # one 3D macro element: 8 points, the other law and coupling: far fewer points than SMs
        dict(name="rve3d_8x8_svk_kubc", kind="rve3d", n_qp=8, sizes="8", precision="mixed", law=1, bc=1),
        # a chunk of the surrogate's training data: the 12^3 two-sphere RVE, no tangent
        dict(name="training_256x12", kind="training", n_qp=256, sizes="12", stages=3),
        # the macro part of the 2D headline and of the 16^3 cantilever
        dict(name="macro_2d_32", kind="macro", dim=2, nx=32, ny=32, nz=1),
        dict(name="macro_3d_16", kind="macro", dim=3, nx=16, ny=16, nz=16),
        # one training step at the batch size of the training loop
        dict(name="mlp_train_4096", kind="mlp", batch=4096),
        # the surrogate at every macro point of the 16^3 cantilever
        dict(name="surrogate_32768", kind="surrogate", n=32768, degree=6),
        # a whole load step of the smallest two-scale problem through the driver: launches, copies and
        # the host loop count
        dict(name="load_step_4x4x8_fp64", kind="step", macro=4, grid=8, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rve2d", "rve2d", "rve2d", "noalloc", "rve3d", "rve3d", "training", "macro", "macro", "mlp",
                       "surrogate", "surrogate", "step"])
    if kind == "rve2d":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        sizes = sorted(rng.sample(range(4, 33, 2), rng.choice([1, 1, 1, 2, 3, 5])))
        return dict(kind=kind, n_qp=_log_int(rng, 4, 2000 if precision == "mixed" else 300),
                    sizes=",".join(map(str, sizes)), precision=precision, law=rng.choice([0, 0, 0, 1]),
                    bc=rng.choice([0, 0, 0, 1]), shared=False)
    if kind == "noalloc":
        return dict(kind=kind, n_qp=_log_int(rng, 1, 200), sizes=str(rng.choice([2, 4, 6, 8, 10, 12, 14, 16])))
    if kind == "rve3d":
        sizes = sorted(rng.sample([4, 5, 6, 7, 8, 10, 12, 14, 16], rng.choice([1, 1, 2, 3])))
        return dict(kind=kind, n_qp=_log_int(rng, 2, 200), sizes=",".join(map(str, sizes)), precision="mixed",
                    law=rng.choice([0, 0, 1]), bc=rng.choice([0, 0, 1]))
    if kind == "training":
        return dict(kind=kind, n_qp=_log_int(rng, 8, 256), sizes=str(rng.choice([6, 8, 12])), stages=rng.choice([1, 2, 3]))
    if kind == "macro":
        if rng.random() < 0.5:
            return dict(kind=kind, dim=2, nx=_log_int(rng, 2, 96), ny=_log_int(rng, 2, 96), nz=1)
        return dict(kind=kind, dim=3, nx=_log_int(rng, 2, 16), ny=_log_int(rng, 2, 16), nz=_log_int(rng, 2, 16))
    if kind == "mlp":
        return dict(kind=kind, batch=_log_int(rng, 64, 16384))
    if kind == "surrogate":
        return dict(kind=kind, n=_log_int(rng, 1, 32768), degree=rng.choice([0, 3, 4, 5, 6, 6]))
    return dict(kind="step", macro=rng.choice([2, 3, 5, 6, 7, 8]), grid=rng.choice([4, 6, 8, 10, 12, 16]),
                precision=rng.choice(["fp64", "mixed"]))


# ------------------------------------------------------------------------------------ inputs
def _phase(n, dim, centers, radius):
    """0 = matrix, 1 = inclusion (periodic balls of one radius), element order x fastest."""
    c1 = (np.arange(n) + 0.5) / n
    inside = np.zeros((n,) * dim, dtype=bool)
    for c in centers:
        r2 = np.zeros((n,) * dim)
        for k in range(dim):
            dk = c1 - c[k]
            dk -= np.round(dk)
            r2 += (dk * dk).reshape([-1 if a == dim - 1 - k else 1 for a in range(dim)])
        inside |= r2 <= radius * radius
    return inside.astype(np.uint8).reshape(-1)


def _rve_inputs(case, seed):
    """Microstructures, materials, and the deformation gradients of this and of the previous load step."""
    r = np.random.default_rng([seed, 11])
    dim = 3 if case["kind"] in ("rve3d", "training") else 2
    sizes = [int(s) for s in case["sizes"].split(",")]
    n_qp = case["n_qp"]
    n_rve = 1 if case.get("shared") or case["kind"] == "training" else n_qp
    n = np.random.default_rng(n_rve).permutation(np.resize(sizes, n_rve)).astype(np.int32)  # the same of every seed
    phases, E = [], np.ones((n_rve, 2))
    for q in range(n_rve):
        if dim == 2:
            phases.append(_phase(int(n[q]), 2, r.random((1, 2)), 0.15 + 0.2 * r.random()))
            E[q, 1] = 10.0 if case.get("shared") else math.exp(r.uniform(math.log(5.0), math.log(50.0)))
        else:
            m = 2 if case["kind"] == "training" else int(r.integers(1, 5))
            vol = r.uniform(0.1, 0.3)
            phases.append(_phase(int(n[q]), 3, r.random((m, 3)), (3.0 * vol / (4.0 * math.pi * m)) ** (1.0 / 3.0)))
            E[q, 1] = 10.0
    qp_rve = (np.arange(n_qp) % n_rve).astype(np.int32)
    eye = np.eye(dim)
    noise = r.uniform(-1.0, 1.0, (n_qp, dim, dim))
    if case["kind"] == "training":  # symmetric stretches uniform in the ball |U - I| <= 0.3
        z = r.standard_normal((n_qp, 6))
        z *= (0.3 * r.random(n_qp) ** (1.0 / 6.0) / np.linalg.norm(z, axis=1))[:, None]
        F1 = np.repeat(eye[None], n_qp, 0)
        for k, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            v = z[:, k] if i == j else z[:, k] / math.sqrt(2.0)
            F1[:, i, j] += v
            if i != j:
                F1[:, j, i] += v
        F0 = F1
    else:  # along a load path of 20 (2D: biaxial and shear) or 10 (3D: uniaxial) steps
        if dim == 2:
            H, dt = np.array([[0.3, 0.3], [0.0, 0.3]]), 1.0 / 20
        else:
            H, dt = np.diag([0.2, -0.05, -0.05]), 1.0 / 10
        if case.get("law"):
            H = 0.5 * H
        t = dt * r.integers(2, round(1 / dt) + 1)
        F1 = eye + t * H + 0.02 * t * noise
        F0 = eye + (t - dt) * (H + 0.02 * noise)
    return dim, n, phases, E, np.full((n_rve, 2), 0.3), qp_rve, F0, F1


def _keep(view, owner):
    """A view of memory that a library object owns keeps that object alive."""
    view.owner = owner
    return view


def _dev(a, dtype=F64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _macro_inputs(case, seed):
    """u of a load step, and the homogenised stress and tangent at every point: a neo-Hookean law whose
    stiffness varies from point to point."""
    d = case["dim"]
    nel = [case["nx"], case["ny"], case["nz"]][:d]
    r = np.random.default_rng([seed, 12])
    n_qp = int(np.prod(nel)) * 2 ** d
    n_node = int(np.prod([m + 1 for m in nel]))
    u = 0.02 * r.standard_normal((n_node, d))
    s = np.exp(r.uniform(0.0, math.log(3.0), n_qp))
    F = np.eye(d) + 0.1 * np.eye(d) + 0.05 * r.uniform(-1, 1, (n_qp, d, d))
    P, A = _law(_dev(F), _dev(0.577 * s), _dev(0.385 * s), 0)
    axes = np.meshgrid(*[np.arange(m + 1) / m for m in nel], indexing="ij")
    X = np.stack([a.transpose().reshape(-1) for a in axes], 1)
    on = np.isclose(X, 0.0).any(1) | np.isclose(X, 1.0).any(1) if d == 2 else np.isclose(X[:, 0], 0.0) | np.isclose(X[:, 0], 1.0)
    nodes = np.nonzero(on)[0]
    dofs = (nodes[:, None] * d + np.arange(d)).reshape(-1)
    vals = 0.1 * X[nodes].reshape(-1)
    return nel, n_qp, _dev(u.reshape(-1)), P.reshape(n_qp, d * d).contiguous(), A.reshape(n_qp, d ** 4).contiguous(), dofs, vals


def _net(seed):
    """Network parameters as after some training: He-scaled weights, small biases."""
    r = np.random.default_rng([seed, 13])
    p = {}
    for l, fan in enumerate([6, 128, 128, 128]):
        p[f"W{l + 1}"] = math.sqrt(6.0 / fan) * r.uniform(-1, 1, (128, fan))
        p[f"b{l + 1}"] = 0.1 * r.uniform(-1, 1, 128)
    p["w5"] = math.sqrt(3.0 / 128) * r.uniform(-1, 1, 128)
    p["b5"] = 0.1 * r.uniform(-1, 1, 1)
    return {k: v.astype(np.float32).astype(np.float64) for k, v in p.items()}


def _mlp_inputs(case, seed):
    r = np.random.default_rng([seed, 14])
    B = case["batch"]
    x = r.uniform(-0.9, 0.9, (B, 6))
    ty = 0.3 * np.sin(x @ r.standard_normal(6)) + 0.2 * (x * x).sum(1)
    tg = 0.4 * x + 0.3 * r.standard_normal((B, 6))
    f = np.float32
    return x.astype(f), ty.astype(f), tg.astype(f), 1.0 / float((ty ** 2).mean()) / B, 1.0 / float((tg ** 2).sum(1).mean()) / B


def _surrogate_inputs(case, seed):
    """Macro deformation gradients (some outside the trust region) and a trained surrogate's parameters."""
    r = np.random.default_rng([seed, 15])
    n = case["n"]
    z = r.standard_normal((n, 9))
    z *= (0.33 * r.random(n) ** (1.0 / 9.0) / np.linalg.norm(z, axis=1))[:, None]
    F = np.eye(3).reshape(1, 9) + z
    Ca = r.standard_normal((6, 6))
    counts = {3: 56, 4: 126, 5: 252, 6: 462}
    poly = np.concatenate([(0.5 ** (d - 3) * r.standard_normal(c)) if d <= case["degree"] else np.zeros(c)
                           for d, c in counts.items()])
    return F, dict(lam0=0.75, mu0=0.5, sx=0.35, sg=0.0175, radius=0.3, Ca=0.01 * (Ca + Ca.T), y0=0.1 * r.standard_normal(),
                   g0=0.1 * r.standard_normal(6), poly=poly)


def _step_problem(case, seed):
    """Uniaxial stretch of a square with symmetry rollers; one circular inclusion."""
    r = np.random.default_rng([seed, 16])
    m, n = case["macro"], case["grid"]
    ax = np.arange(m + 1) / m
    X = np.stack([np.tile(ax, m + 1), np.repeat(ax, m + 1)], 1)
    dofs = np.concatenate([np.nonzero(X[:, a] == 0.0)[0] * 2 + a for a in (0, 1)] + [np.nonzero(X[:, 0] == 1.0)[0] * 2])
    vals = np.concatenate([np.zeros(2 * (m + 1)), np.full(m + 1, 0.1)])
    order = np.argsort(dofs, kind="stable")
    return SimpleNamespace(dim=2, macro_n=(m, m), rve_n=np.array([n]), rve_phase=[_phase(n, 2, r.random((1, 2)), 0.25)],
                           rve_E=np.array([[1.0, 10.0]]), rve_nu=np.array([[0.3, 0.3]]),
                           qp_rve=np.zeros(4 * m * m, dtype=np.int64), n_qp=4 * m * m, dirichlet_dofs=dofs[order],
                           dirichlet_end=vals[order], n_steps=10, precision=case["precision"], newton_tol=1e-10)


# ------------------------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case)
    if kind in ("rve2d", "rve3d", "training"):
        dim, n, phases, E, nu, qp_rve, F0, F1 = _rve_inputs(case, seed)
        s.ctx = fe.Context(dim, case.get("precision", "mixed"), law=case.get("law", 0), bc=case.get("bc", 0))
        s.ctx.add_rves(n, phases, E, nu)
        s.ctx.bind_qps(qp_rve)
        s.F = _dev(F1.reshape(-1, dim * dim))
        s.P, s.A = torch.zeros_like(s.F), torch.zeros(len(F1), dim ** 4, dtype=F64, device="cuda")
        s.st = torch.zeros(len(F1), dtype=I32, device="cuda")
        s.w = _keep(s.ctx.fluctuations(), s.ctx)
        if kind != "training":  # the converged state of the previous load step
            s.ctx.rve_solve(_dev(F0.reshape(-1, dim * dim)), s.P, s.A, s.st)
            s.ctx.commit()
    elif kind == "noalloc":
        _, n, phases, E, nu, _, F0, F1 = _rve_inputs(case, seed)
        lame = np.zeros((len(n), 4, 2))
        lame[:, :2, 0] = E * nu / ((1 + nu) * (1 - 2 * nu))
        lame[:, :2, 1] = E / (2 * (1 + nu))
        s.n, s.n_qp = int(n[0]), case["n_qp"]
        s.phase, s.lame = _dev(np.stack(phases), torch.uint8), _dev(lame)
        s.F, s.w = _dev(F1.reshape(-1, 4)), torch.zeros(s.n_qp, 2 * s.n * s.n, dtype=F64, device="cuda")
        s.P, s.A = torch.zeros(s.n_qp, 4, dtype=F64, device="cuda"), torch.zeros(s.n_qp, 16, dtype=F64, device="cuda")
        s.st = torch.zeros(s.n_qp, dtype=I32, device="cuda")
        s.opt = fe.Options()
        fe.lib().fehmm_default_options(ctypes.byref(s.opt), 2, fe.PREC_FP64)
        _noalloc(s, _dev(F0.reshape(-1, 4)))
        s.w0 = s.w.clone()
    elif kind == "macro":
        nel, n_qp, s.u, s.P, s.A, dofs, vals = _macro_inputs(case, seed)
        d = case["dim"]
        s.ctx = fe.Context(d, "mixed")
        s.ctx.macro_create(nel)
        s.ctx.macro_set_dirichlet(dofs, vals)
        _, _, rows, nnz = s.ctx.macro_csr()
        s.F = torch.zeros(n_qp, d * d, dtype=F64, device="cuda")
        s.f, s.du, s.info = (torch.zeros(m, dtype=F64, device="cuda") for m in (rows, rows, 3))
        s.K = torch.zeros(nnz, dtype=F64, device="cuda")
    elif kind == "mlp":
        x, ty, tg, s.cy, s.cg = _mlp_inputs(case, seed)
        s.x, s.ty, s.tg = _dev(x, F32), _dev(ty, F32), _dev(tg, F32)
        s.loss = torch.zeros(1, dtype=F32, device="cuda")
        s.mlp = su.MLP(case["batch"])
        s.mlp.set_params(_net(seed))
        s.grad = _keep(s.mlp.grad_buffer(), s.mlp)
    elif kind == "surrogate":
        F, p = _surrogate_inputs(case, seed)
        n = case["n"]
        s.F = _dev(F)
        s.P, s.A = torch.zeros(n, 9, dtype=F64, device="cuda"), torch.zeros(n, 81, dtype=F64, device="cuda")
        s.W, s.inside = torch.zeros(n, dtype=F64, device="cuda"), torch.zeros(n, dtype=I32, device="cuda")
        s.work = torch.zeros(su.work_floats(n), dtype=F32, device="cuda")
        s.mlp = su.MLP(n)
        s.mlp.set_params(_net(seed))
        s.sp = su.SurrogateParams(p["lam0"], p["mu0"], p["sx"], p["sg"], p["radius"])
        s.sp.set_Ca(p["Ca"])
        s.sp.y0 = p["y0"]
        s.sp.g0[:] = p["g0"].tolist()
        s.sp.poly[:] = p["poly"].tolist()
    else:
        s.drv = LoadStepDriver(_step_problem(case, seed))
        s.drv.load_step(1)
        s.state = s.drv.state()
        s.w = _keep(s.drv.ctx.fluctuations(), s.drv.ctx)
    return s


def _noalloc(s, F):
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = fe.lib().fehmm_rve2d_solve_fp64_noalloc(s.n_qp, s.n, 1, ptr(s.phase), ptr(s.lame), ptr(s.w), ptr(F), ptr(s.P),
                                                 ptr(s.A), ptr(s.st), None, ctypes.byref(s.opt),
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc != 0:
        raise fe.FehmmError(fe.status_str(rc))


def run(s):
    kind = s.case["kind"]
    if kind in ("rve2d", "rve3d"):
        s.ctx.rve_solve(s.F, s.P, s.A, s.st, flags=fe.SOLVE_FROM_COMMITTED)
        return {"P": s.P, "A": s.A, "status": s.st, "w": s.w}
    if kind == "training":
        P, _, W, st = su.rve_solve_batch(s.ctx, s.F, stages=s.case["stages"])
        return {"P": P, "W": W, "status": st, "w": s.w}
    if kind == "noalloc":
        s.w.copy_(s.w0)  # the entry updates the caller's fluctuations in place
        _noalloc(s, s.F)
        return {"P": s.P, "A": s.A, "status": s.st, "w": s.w}
    if kind == "macro":
        s.ctx.macro_qp_F(s.u, s.F)
        s.ctx.macro_assemble(s.P, s.A, s.f, s.K)
        s.ctx.macro_solve(s.K, s.f, s.du, s.info)
        # of info, |f_free| (what convergence is judged by); the CG's iteration count is a diagnostic
        return {"F": s.F, "f": s.f, "K": s.K, "du": s.du, "norm": s.info[:1]}
    if kind == "mlp":
        s.mlp.loss_grad(s.x, s.ty, s.tg, s.cy, s.cg, s.loss)
        s.mlp.adamw(1e-3)
        return {"loss": s.loss, "grad": s.grad}
    if kind == "surrogate":
        su.surrogate_eval(s.mlp, s.sp, s.F, s.P, s.A, s.W, s.inside, s.work)
        return {"P": s.P, "A": s.A, "W": s.W, "inside": s.inside}
    s.drv.restore(s.state)
    rec = s.drv.load_step(2, commit=False)
    return {"u": s.drv.u, "P": s.drv.P, "A": s.drv.A, "w": s.w, "converged": rec["converged"]}


# ------------------------------------------------------------------------------------ work
def work(case):
    """Bytes: each input read once, each output and updated state written once. Operations: of an RVE
    solve, what three Newton corrections and the transfer of a multigrid-preconditioned solver cannot do
    without: residuals, tangents and ten operator products a linear solve; of the rest, of the formulas."""
    kind = case["kind"]
    if kind in ("rve2d", "rve3d", "training", "noalloc"):
        d = 3 if kind in ("rve3d", "training") else 2
        sizes = [int(v) for v in case["sizes"].split(",")]
        el = case["n_qp"] * sum(n ** d for n in sizes) / len(sizes)
        tangent = kind != "training"
        stages = case.get("stages", 1)
        state = 2 * 8 * d * el  # fluctuations in and out
        if tangent and kind != "noalloc":  # kept transfer solutions in and out
            state += 2 * (4 if case["precision"] == "mixed" else 8) * d ** 3 * el
        io = case["n_qp"] * 8 * (2 * d * d + (d ** 4 if tangent else 1))
        residual, stiff, product = (200, 1300, 100) if d == 2 else (2600, 4200, 4000)
        solves = 3 * stages + (d * d if tangent else 0)
        return {"bytes": state + io + el, "flops": el * (stages * (4 * residual + 4 * stiff) + 10 * solves * product)}
    if kind == "macro":
        d = case["dim"]
        nel = [case["nx"], case["ny"], case["nz"]][:d]
        qp, nodes = np.prod(nel) * 2 ** d, np.prod([m + 1 for m in nel])
        nnz = np.prod([3 * m + 1 for m in nel]) * d * d
        # one CG iteration per node layer at least: the correction has to cross the mesh
        its = max(nel)
        return {"bytes": float(8 * (qp * (2 * d * d + d ** 4) + nodes * d * 3 + nnz)),
                "flops": float(qp * 4 ** d * 4 * d ** 4 + its * 2 * nnz)}
    if kind == "mlp":
        B = case["batch"]
        # forward, input gradient, and back through both: 12 layer products and 6 of the weight gradients
        return {"bytes": 4.0 * (B * 13 + 5 * 51205), "flops": B * 18.0 * 2 * 128 * 128}
    if kind == "surrogate":
        n = case["n"]
        # the network's value, gradient and six tangent directions (bf16); the polynomial's Hessian (FP64)
        return {"bytes": n * (8.0 * (9 + 9 + 81 + 1) + 4), "flops": n * (7 * 6 * 2 * 128 * 128 + 2 * 21 * 209.0)}
    m, n = case["macro"], case["grid"]
    el = 4 * m * m * n * n
    return {"bytes": 3.0 * (2 * 8 * 2 * el + 2 * 8 * 8 * el), "flops": 3.0 * el * (4 * 200 + 4 * 1300 + 10 * 7 * 100)}


# ------------------------------------------------------------------------------------ exact
def _law(F, lam, mu, law):
    """First Piola-Kirchhoff stress and dP/dF (batch x d x d, batch x d x d x d x d)."""
    d = F.shape[-1]
    eye = torch.eye(d, dtype=F.dtype, device=F.device)
    lam_, mu_ = lam[:, None, None], mu[:, None, None]
    L4, M4 = lam[:, None, None, None, None], mu[:, None, None, None, None]
    if law == 0:  # neo-Hooke: P = mu F + hb F^-T
        J = torch.linalg.det(F)[:, None, None]
        Fit = torch.linalg.inv(F).transpose(1, 2)
        hb, gm = 0.5 * lam_ * (J * J - 1) - mu_, lam_ * J * J
        P = mu_ * F + hb * Fit
        A = (M4 * torch.einsum("ik,jl->ijkl", eye, eye) - hb[..., None, None] * torch.einsum("qil,qkj->qijkl", Fit, Fit)
             + gm[..., None, None] * torch.einsum("qij,qkl->qijkl", Fit, Fit))
        return P, A
    E = 0.5 * (F.transpose(1, 2) @ F - eye)
    S = lam_ * E.diagonal(dim1=1, dim2=2).sum(1)[:, None, None] * eye + 2 * mu_ * E
    b = F @ F.transpose(1, 2)
    A = (torch.einsum("ik,qjl->qijkl", eye, S) + L4 * torch.einsum("qij,qkl->qijkl", F, F)
         + M4 * (torch.einsum("qik,jl->qijkl", b, eye) + torch.einsum("qil,qkj->qijkl", F, F)))
    return F @ S, A


def _shape_grads(d):
    """dN_a/dxi_J at the Gauss points of [0,1]^d (corner a = bits x, y, z) -> [q, a, J]."""
    g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    G = np.zeros((2 ** d, 2 ** d, d))
    for q in range(2 ** d):
        for a in range(2 ** d):
            for J in range(d):
                v = 1.0 if (a >> J) & 1 else -1.0
                for k in range(d):
                    if k != J:
                        t = g[(q >> k) & 1]
                        v *= t if (a >> k) & 1 else 1 - t
                G[q, a, J] = v
    return G


def _rve_exact(n, d, phase, E, nu, F, law, bc, tangent):
    """P, A, W and w of RVEs of one grid size (batched, dense Newton in 64 bits)."""
    B, NN, D = len(F), n ** d, d * n ** d
    idx = np.indices((n,) * d).reshape(d, -1)[::-1]  # x fastest
    conn = np.stack([sum((((idx[k] + ((a >> k) & 1)) % n) * n ** k) for k in range(d)) for a in range(2 ** d)], 1)
    pinned = (idx == 0).any(0) if bc else (np.arange(NN) == 0)
    free = torch.tensor(np.repeat(~pinned, d), device="cuda")
    G = _dev(_shape_grads(d) * n)
    conn = torch.tensor(conn, device="cuda")
    dof = (conn[:, :, None] * d + torch.arange(d, device="cuda")).reshape(NN, -1)
    lam = _dev(np.take_along_axis(E * nu / ((1 + nu) * (1 - 2 * nu)), phase.astype(int), 1))
    mu = _dev(np.take_along_axis(E / (2 * (1 + nu)), phase.astype(int), 1))
    wq, NQ = 1.0 / (2 ** d * NN), 2 ** d
    lq, mq = (v[:, :, None].expand(B, NN, NQ).reshape(-1) for v in (lam, mu))
    Fb = _dev(F)
    w = torch.zeros(B, NN, d, dtype=F64, device="cuda")

    def state(Ft):
        Fq = Ft[:, None, None] + torch.einsum("beai,qaj->beqij", w[:, conn], G)
        P, A = _law(Fq.reshape(-1, d, d), lq, mq, law)
        return Fq, P.reshape(B, NN, NQ, d, d), A.reshape(B, NN, NQ, d, d, d, d)

    def matrix(A):
        Ke = wq * torch.einsum("qaj,beqijkl,qcl->beaick", G, A, G).reshape(B, NN, -1)
        K = torch.zeros(B, D * D, dtype=F64, device="cuda")
        at = (dof[:, :, None] * D + dof[:, None, :]).reshape(-1)
        K.index_add_(1, at, Ke.reshape(B, -1))
        K = K.reshape(B, D, D) * free[:, None] * free[None, :]
        return K + torch.diag((~free).to(F64))

    eye = torch.eye(d, dtype=F64, device="cuda")
    for stage in range(1, 3):  # half the load first
        Ft = eye + (Fb - eye) * (stage / 2)
        for _ in range(12):
            _, P, A = state(Ft)
            R = torch.zeros(B, D, dtype=F64, device="cuda")
            R.index_add_(1, dof.reshape(-1), wq * torch.einsum("beqij,qaj->beai", P, G).reshape(B, -1))
            R *= free
            if float(R.abs().max()) < 1e-16 * (1 if stage == 2 else 1e6):
                break
            dw = torch.linalg.solve(matrix(A), -R)
            w += dw.reshape(B, NN, d)
            if float(dw.abs().max()) < (1e-14 if stage == 2 else 1e-6):
                break
    Fq, P, A = state(Fb)
    out = {"P": wq * P.sum((1, 2)).reshape(B, -1), "w": w.reshape(B, -1), "A": None}
    C = Fq.transpose(-1, -2) @ Fq
    lb, mb = lam[:, :, None], mu[:, :, None]
    if law == 0:
        J = torch.linalg.det(Fq)
        W = 0.25 * lb * (J * J - 1) - (0.5 * lb + mb) * J.log() + 0.5 * mb * (C.diagonal(dim1=-2, dim2=-1).sum(-1) - d)
    else:
        Eg = 0.5 * (C - eye)
        W = 0.5 * lb * Eg.diagonal(dim1=-2, dim2=-1).sum(-1) ** 2 + mb * (Eg * Eg).sum((-1, -2))
    out["W"] = wq * W.sum((1, 2))
    if tangent:
        L = torch.zeros(B, D, d * d, dtype=F64, device="cuda")
        L.index_add_(1, dof.reshape(-1), wq * torch.einsum("qaj,beqijkl->beaikl", G, A).reshape(B, -1, d * d))
        L *= free[:, None]
        X = torch.linalg.solve(matrix(A), -L)
        out["A"] = (wq * A.sum((1, 2)).reshape(B, d * d, d * d) + L.transpose(1, 2) @ X).reshape(B, -1)
    return out


def _exact_rves(case, seed):
    dim, n, phases, E, nu, qp_rve, _, F1 = _rve_inputs(case, seed)
    if sum((dim * float(n[r]) ** dim) ** 3 * 8 for r in qp_rve) > 6e12:  # dense factorisations: beyond some seconds
        return None
    tangent, law, bc = case["kind"] != "training", case.get("law", 0), case.get("bc", 0)
    parts, keys = {}, ("P", "A", "W", "w") if tangent else ("P", "W", "w")
    for size in sorted(set(n.tolist())):
        qps = np.nonzero(n[qp_rve] == size)[0]
        step = max(1, int(2e9 // (8 * (dim * size ** dim) ** 2 + 8 * size ** dim * 2 ** dim * dim ** 4)))
        for at in range(0, len(qps), step):
            q = qps[at:at + step]
            r = qp_rve[q]
            o = _rve_exact(size, dim, np.stack([phases[k] for k in r]), E[r], nu[r], F1[q], law, bc, tangent)
            for k in keys:
                for i, p in enumerate(q):
                    parts.setdefault(k, {})[p] = o[k][i]
    out = {k: torch.stack([v[p] for p in range(len(F1))]) if k != "w" else torch.cat([v[p] for p in range(len(F1))])
           for k, v in parts.items()}
    if case["kind"] == "noalloc":
        out["w"] = out["w"].reshape(len(F1), -1)
    if tangent:
        out.pop("W")
    return {**out, "status": None}


def _exact_macro(case, seed):
    nel, n_qp, u, P, A, dofs, _ = _macro_inputs(case, seed)
    d, ne, N = case["dim"], int(np.prod(nel)), [m + 1 for m in nel]
    el = np.stack(np.unravel_index(np.arange(ne), nel[::-1])[::-1], 1)  # x fastest
    corner = [[(a >> k) & 1 for k in range(d)] for a in range(2 ** d)]
    stride = np.cumprod([1] + N[:-1])
    pos = np.stack([el + np.array(c) for c in corner], 1)  # [ne, a, d]
    node = torch.tensor(pos @ stride, device="cuda")
    G = _dev(_shape_grads(d) * np.array(nel, dtype=float))  # [q, a, J]
    om = 1.0 / n_qp
    ue = u.reshape(-1, d)[node]
    F = torch.eye(d, dtype=F64, device="cuda") + torch.einsum("eai,qaj->eqij", ue, G)
    n_node = int(np.prod(N))
    f = torch.zeros(n_node, d, dtype=F64, device="cuda")
    f.index_add_(0, node.reshape(-1), om * torch.einsum("eqij,qaj->eai", P.reshape(ne, -1, d, d), G).reshape(-1, d))
    Ke = om * torch.einsum("qaj,eqijkl,qcl->eaick", G, A.reshape(ne, -1, d, d, d, d), G)
    # CSR: rows node-major, of each node its neighbours (clipped 3^d box) in order, d columns each
    X = np.stack(np.unravel_index(np.arange(n_node), N[::-1])[::-1], 1)
    lo, hi = np.maximum(X - 1, 0), np.minimum(X + 1, np.array(N) - 1)
    box = hi - lo + 1
    deg = box.prod(1)
    rowptr = np.concatenate([[0], np.cumsum(np.repeat(deg * d, d))])
    mul = np.concatenate([np.ones((n_node, 1), int), np.cumprod(box, 1)[:, :-1]], 1)
    nd = pos @ stride
    at = np.zeros((ne, 2 ** d, d, 2 ** d, d), dtype=np.int64)
    col = np.zeros(rowptr[-1], dtype=np.int64)
    for a in range(2 ** d):
        for c in range(2 ** d):
            I = nd[:, a]
            rank = ((pos[:, c] - lo[I]) * mul[I]).sum(1)
            for i in range(d):
                for k in range(d):
                    at[:, a, i, c, k] = rowptr[I * d + i] + rank * d + k
                    col[at[:, a, i, c, k]] = nd[:, c] * d + k
    K = torch.zeros(int(rowptr[-1]), dtype=F64, device="cuda")
    K.index_add_(0, torch.tensor(at.reshape(-1), device="cuda"), Ke.reshape(-1))
    free = torch.ones(n_node * d, dtype=F64, device="cuda")
    free[torch.tensor(dofs, device="cuda")] = 0.0
    f = f.reshape(-1)
    row = np.repeat(np.arange(n_node * d), np.diff(rowptr))
    rt, ct = torch.tensor(row, device="cuda"), torch.tensor(col, device="cuda")
    diag = torch.ones(n_node * d, dtype=F64, device="cuda").index_copy_(0, rt[rt == ct], K[rt == ct])
    M = torch.sparse_csr_tensor(torch.tensor(rowptr, device="cuda"), ct, K, (n_node * d, n_node * d))
    x, b = torch.zeros_like(f), -f * free
    for _ in range(2):  # Jacobi-CG to rounding, and once more on what it left
        r = b - (M @ x) * free
        z = r / diag
        p, rz, first = z.clone(), float(r @ z), None
        first = rz
        for _it in range(20 * int(math.sqrt(n_node * d)) + 200):
            if not rz > 1e-31 * first:
                break
            q = (M @ p) * free
            al = rz / float(p @ q)
            x += al * p
            r -= al * q
            z = r / diag
            new = float(r @ z)
            p, rz = z + (new / rz) * p, new
    return {"F": F.reshape(n_qp, -1), "f": f, "K": K, "du": x, "norm": (f * free).norm().reshape(1)}


def _forward(p, x):
    a = x
    for l in range(1, 5):
        a = torch.nn.functional.silu(a @ p[f"W{l}"].T + p[f"b{l}"])
    return a @ p["w5"] + p["b5"]


def _exact_mlp(case, seed):
    x, ty, tg, cy, cg = _mlp_inputs(case, seed)
    p = {k: _dev(v).requires_grad_() for k, v in _net(seed).items()}
    xt = _dev(x).requires_grad_()
    y = _forward(p, xt)
    (g,) = torch.autograd.grad(y.sum(), xt, create_graph=True)
    loss = 0.5 * (cy * (y - _dev(ty)) ** 2).sum() + 0.5 * cg * ((g - _dev(tg)) ** 2).sum()
    gr = dict(zip(p, torch.autograd.grad(loss, list(p.values()))))
    W1 = torch.zeros(128, 8, dtype=F64, device="cuda")
    W1[:, :6] = gr["W1"]
    parts = [W1, gr["b1"]] + [gr[k] for l in (2, 3, 4) for k in (f"W{l}", f"b{l}")] + [gr["w5"], gr["b5"],
                                                                                      torch.zeros(3, dtype=F64, device="cuda")]
    return {"loss": loss.detach().reshape(1), "grad": torch.cat([v.detach().reshape(-1) for v in parts])}


def _exact_surrogate(case, seed):
    Fh, s = _surrogate_inputs(case, seed)
    p = {k: _dev(v) for k, v in _net(seed).items()}
    mono, c0 = [], 0
    for d in range(3, 7):
        tup = [()]
        for _ in range(d):
            tup = [t + (k,) for t in tup for k in range(t[-1] if t else 0, 6)]
        if s["poly"][c0:c0 + len(tup)].any():
            mono.append((torch.tensor(tup, device="cuda"), _dev(s["poly"][c0:c0 + len(tup)])))
        c0 += len(tup)
    I6, J6 = [0, 1, 2, 1, 0, 0], [0, 1, 2, 2, 2, 1]
    wt = _dev(np.array([1.0, 1, 1] + [math.sqrt(2.0)] * 3))
    Ca, g0 = _dev(s["Ca"]), _dev(s["g0"])
    Ps, As, Ws = [], [], []
    for part in _dev(Fh).split(4096):
        F = part.clone().requires_grad_()
        F3 = F.reshape(-1, 3, 3)
        C = F3.transpose(1, 2) @ F3
        m = 0.5 * wt * (C - torch.eye(3, dtype=F64, device="cuda"))[:, I6, J6]
        J2 = torch.linalg.det(C)
        W = (0.25 * s["lam0"] * (J2 - 1) - (0.5 * s["lam0"] + s["mu0"]) * 0.5 * J2.log()
             + 0.5 * s["mu0"] * (C.diagonal(dim1=1, dim2=2).sum(1) - 3) + 0.5 * ((m @ Ca) * m).sum(1))
        x = m / s["sx"]
        y = _forward(p, x) - s["y0"] - x @ g0
        for tup, coef in mono:
            y = y + torch.stack([x[:, tup[:, k]] for k in range(tup.shape[1])]).prod(0) @ coef
        W = W + s["sg"] * y
        (P,) = torch.autograd.grad(W.sum(), F, create_graph=True)
        A = torch.stack([torch.autograd.grad(P[:, k].sum(), F, retain_graph=True)[0] for k in range(9)], 1)
        Ps.append(P.detach())
        As.append(A.reshape(-1, 81))
        Ws.append(W.detach())
    return {"P": torch.cat(Ps), "A": torch.cat(As), "W": torch.cat(Ws), "inside": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("rve2d", "rve3d", "training", "noalloc"):
        return _exact_rves(case, seed)
    if kind == "macro":
        return _exact_macro(case, seed)
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "surrogate":
        return _exact_surrogate(case, seed)
    return None  # a whole load step: many solves deep
