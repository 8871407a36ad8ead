"""A macro solve that gives up (info status 3: its correction is not valid) ends a load step, a tangent predictor and a
sharded iteration with an error, on every rank and before the correction is used.  The context is a stand-in on the
CPU whose macro solve reports the status; everything else is the package's own host code."""
import os

import numpy as np
import pytest
import torch

from paper_1908_08292_gb300 import FehmmError
from paper_1908_08292_gb300.dist import Shard, ShardedIteration
from paper_1908_08292_gb300.driver import LoadStepDriver
from test_dist_gloo import _free_port


class StandIn:
    """Records the calls; macro solve number `fails` (from 1) gives up, the others converge to |f| = norm."""

    def __init__(self, fails=0, norm=1e-30):
        self.fails, self.norm, self.solves, self.calls = fails, norm, 0, []

    def macro_solve(self, K, f, du, info, rtol=0.0):
        self.solves += 1
        self.calls.append("solve")
        info.copy_(torch.tensor([np.nan, 5.0, 3.0] if self.solves == self.fails else [self.norm, 5.0, 0.0]))

    def __getattr__(self, name):
        return lambda *a, **k: self.calls.append(name)


def driver(ctx, predictor):
    d = object.__new__(LoadStepDriver)
    z = lambda *n: torch.zeros(*n, dtype=torch.float64)  # noqa: E731
    d.p = type("Problem", (), {"n_steps": 10})()
    d.ctx, d.scheme, d.predictor, d.K_valid, d.scale, d.graphs, d.shard = ctx, "nested", predictor, True, 0.0, False, None
    d.macro_rtol, d.macro_atol, d.max_macro, d.solve_rtol = 1e-10, 1e-13, 4, 1e-12
    d.u, d.du, d.f, d.g, d.K, d.info, d.F, d.P, d.A = z(8), z(8), z(8), z(8), z(64), z(3), z(4, 4), z(4, 4), z(4, 16)
    d.st, d.it = torch.zeros(4, dtype=torch.int32), torch.zeros(4, 4, dtype=torch.int32)
    d.rve_events = d.iter_log = None
    return d


# without predictor the first solve belongs to the first macro iteration, with it to the predictor; a norm above the
# tolerance lets a second iteration follow
@pytest.mark.parametrize("predictor,fails,norm", [(False, 1, 1e-30), (False, 2, 1.0), (True, 1, 1e-30), (True, 2, 1e-30)])
def test_load_step_raises(predictor, fails, norm):
    ctx = StandIn(fails, norm)
    d = driver(ctx, predictor)
    with pytest.raises(FehmmError, match="gave up"):
        d.load_step(1)
    assert ctx.solves == fails and ctx.calls[-1] == "solve"  # nothing after it: neither its correction nor a commit


def _rank(rank, port, out):
    import torch.distributed as dist
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port))
    dist.init_process_group("gloo", rank=rank, world_size=2)
    try:
        it = object.__new__(ShardedIteration)
        it.ctx, it.shard = StandIn(fails=2), Shard(rank, 2, rank, rank + 1, 4)
        it.P = it.A = None
        it.f, it.K, it.du, it.info = (torch.zeros(n, dtype=torch.float64) for n in (8, 64, 8, 3))
        it.assemble_and_solve()
        try:
            it.assemble_and_solve()
            text = "no error"
        except FehmmError as e:
            text = str(e)
        open(os.path.join(out, f"{rank}.txt"), "w").write(text)
    finally:
        dist.destroy_process_group()


def test_sharded_iteration_raises_on_every_rank(tmp_path):
    import torch.multiprocessing as mp
    mp.spawn(_rank, args=(_free_port(), str(tmp_path)), nprocs=2, join=True)
    for rank in range(2):
        assert "gave up" in (tmp_path / f"{rank}.txt").read_text()
