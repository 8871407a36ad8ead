"""Batches of several grid sizes that share a kernel: each size is a launch with shared memory of its own size, forked
from the caller's stream.  From a non-blocking stream, recorded into a graph (and two such graphs replayed in turn), and
from two host threads with a context each, always against the plain call."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# per dimension and precision: sizes whose launches share an instantiation, the largest one's shared memory beyond
# what a kernel has without asking for it
CASES = [(2, "mixed", [20, 4, 30, 10]), (2, "fp64", [8, 16, 6]), (2, "fp64", [18, 22]), (2, "fp64", [24, 32, 28]),
         (3, "mixed", [9, 3, 6]), (3, "fp64", [7, 2, 5])]


def context(dim, precision, sizes, n_qp, seed):
    import paper_1908_08292_gb300 as fe

    u = synth.uniform(seed, np.arange(len(sizes)), 4)
    phases = [synth.phase_from_inclusions(n, dim, [u[k, :dim]], [0.2 + 0.1 * u[k, 3]]) for k, n in enumerate(sizes)]
    ctx = fe.Context(dim, precision)
    ctx.add_rves(sizes, phases, np.tile([1.0, 8.0], (len(sizes), 1)), np.full((len(sizes), 2), 0.3))
    ctx.bind_qps(np.arange(n_qp, dtype=np.int32) % len(sizes))
    return ctx


def buffers(dim, n_qp, seed):
    import torch

    dev = torch.device("cuda:0")
    F = torch.tensor(synth.random_F(seed, n_qp, dim, 0.05).reshape(n_qp, dim * dim), device=dev)
    return (F, torch.zeros(n_qp, dim * dim, dtype=torch.float64, device=dev),
            torch.zeros(n_qp, dim ** 4, dtype=torch.float64, device=dev),
            torch.full((n_qp,), -1, dtype=torch.int32, device=dev))


def solve(ctx, b):
    import paper_1908_08292_gb300 as fe
    b[1].zero_(), b[2].zero_()
    ctx.rve_solve(*b, flags=fe.SOLVE_FROM_COMMITTED)


def same(dim, b, ref):
    """The 3D tangents come from sums in no fixed order (FP32 or FP64 atomics): to rounding; all else bit by bit."""
    for k in (1, 2, 3):
        got, want = b[k].cpu().numpy(), ref[k].cpu().numpy()
        if dim == 3 and k < 3:
            assert np.abs(got - want).max() <= (1e-6 if k == 2 else 1e-9) * np.abs(want).max()
        else:
            np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("dim,precision,sizes", CASES)
def test_stream_and_graph(dim, precision, sizes):
    import torch

    n_qp = 2 * len(sizes) + 1
    with context(dim, precision, sizes, n_qp, 851) as ctx, context(dim, precision, sizes[:1], 2, 852) as one:
        ref, b, small, small_ref = buffers(dim, n_qp, 853), buffers(dim, n_qp, 853), buffers(dim, 2, 854), buffers(dim, 2, 854)
        solve(ctx, ref)
        solve(one, small_ref)
        torch.cuda.synchronize()
        assert int(ref[3].abs().max()) == 0
        s = torch.cuda.Stream()  # does not wait for the legacy stream
        with torch.cuda.stream(s):
            solve(ctx, b)
        s.synchronize()
        same(dim, b, ref)
        g, g_small = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            solve(ctx, b)
        with torch.cuda.graph(g_small):  # the first size alone, between the two replays
            solve(one, small)
        for _ in range(2):
            for t in b[1:3]:
                t.fill_(5.0)
            g.replay()
            g_small.replay()
            torch.cuda.synchronize()
            same(dim, b, ref)
            same(dim, small, small_ref)


@pytest.mark.parametrize("dim,precision,sizes", [(2, "fp64", [6, 16]), (2, "mixed", [2, 30]), (3, "fp64", [2, 16])])
def test_threads_with_a_context_each(dim, precision, sizes):
    """Half of the threads have a grid that needs little shared memory, half one that needs much; all launch one kernel.
    Bursts of short solves (from the converged state, without tangent) with an empty queue in front of them, so that the
    calls of the threads interleave."""
    import torch

    import paper_1908_08292_gb300 as fe

    failed, bursts, threads = [], 40, 6
    torch.cuda.init()
    together = threading.Barrier(threads)

    def work(size, seed):
        torch.cuda.set_device(0)
        with torch.cuda.stream(torch.cuda.Stream()), context(dim, precision, [size], 1, seed) as ctx:
            b = buffers(dim, 1, seed + 1)
            ctx.rve_solve(*b)
            stream = torch.cuda.current_stream()
            args = (ctx._h, b[0].data_ptr(), b[1].data_ptr(), None, None, b[3].data_ptr(), None, fe.SOLVE_NO_TANGENT,
                    stream.cuda_stream)
            call = fe.lib().fehmm_rve_solve
            for _ in range(bursts):
                together.wait()
                failed.append(sum(call(*args) != 0 for _ in range(100)))
                stream.synchronize()
            failed.append(int(b[3][0]))

    t = [threading.Thread(target=work, args=(sizes[k % 2], 860 + 10 * k)) for k in range(threads)]
    [x.start() for x in t]
    [x.join(120) for x in t]
    assert len(failed) == threads * (bursts + 1) and sum(failed) == 0, failed
