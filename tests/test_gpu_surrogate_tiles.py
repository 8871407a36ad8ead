"""Surrogate evaluation of more points than the combine kernel has blocks for: a block then takes several tiles of 32
points with the polynomial's table of the first.  Every point's result must be the one of a call small enough for one
tile per block, bit for bit (the small calls are compared with the oracle elsewhere), with and without the tangent."""
import numpy as np
import pytest

import synth
from test_gpu_mlp import net

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [0, 4, 6])
@pytest.mark.parametrize("tangent", [True, False])
def test_several_tiles_per_block(degree, tangent):
    import torch

    from paper_1908_08292_gb300.surrogate import MLP, SurrogateParams, surrogate_eval, work_floats
    dev = torch.device("cuda:0")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * 2 * sms * 32 + 32 + 13  # two tiles for every block, a third for one, and a partial one
    F = torch.tensor(synth.random_F(91, n, 3, 0.2), dtype=torch.float64, device=dev).reshape(n, 9)
    m = MLP(n)
    m.set_params(net(92))
    sp = SurrogateParams(1.5, 0.9, 0.35, 0.02, 0.3)
    M = synth.random_field(93, 6, 6, 0.1)
    sp.set_Ca(M + M.T)
    terms = {0: 0, 4: 182, 6: 896}[degree]
    sp.poly[:] = np.concatenate([synth.random_field(94, 1, 896, 0.3)[0][:terms], np.zeros(896 - terms)]).tolist()

    def evaluate(f):
        k = f.shape[0]
        P, A = torch.zeros(k, 9, dtype=torch.float64, device=dev), torch.zeros(k, 81, dtype=torch.float64, device=dev)
        W, ins = torch.zeros(k, dtype=torch.float64, device=dev), torch.zeros(k, dtype=torch.int32, device=dev)
        work = torch.zeros(work_floats(k), device=dev)
        surrogate_eval(m, sp, f.contiguous(), P, A if tangent else None, W, ins, work)
        torch.cuda.synchronize()
        return P, A, W, ins

    whole = evaluate(F)
    step = 32 * sms
    parts = [evaluate(F[a:a + step]) for a in range(0, n, step)]
    for k in range(4):
        got, ref = whole[k], torch.cat([p[k] for p in parts])
        assert torch.equal(got, ref), k
    assert bool(torch.isfinite(whole[0]).all()) and float(whole[0].abs().max()) > 0
    m.close()
