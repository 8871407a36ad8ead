"""The whole-network kernels of the surrogate MLP at the edges of their tiles: 16 samples (value, gradient and
Hessian), 32, 64 or 128 samples (gradient; loss gradient) by the batch's size, and several tiles per block.
Against the oracle network with the operands of every product rounded to bfloat16: what remains is FP32
summation order, within a few bfloat16 units (2^-8)."""
import numpy as np
import pytest

import synth
from oracle import mlp as omlp
from oracle import surrogate as osur
from test_gpu_mlp import net, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 33, 4864, 4865, 9729, 19500])
def test_loss_gradient_every_tile_size(B):
    import torch

    from paper_1908_08292_gb300.surrogate import MLP, unpack
    p = net(71)
    x = synth.random_field(72, B, 6, 0.9).astype(np.float32)
    ty = synth.random_field(73, 1, B, 1.0)[0].astype(np.float32)
    tg = synth.random_field(74, B, 6, 1.0).astype(np.float32)
    cy, cg = 0.7 / B, 1.3 / B
    dev = torch.device("cuda:0")
    m = MLP(B)
    m.set_params(p)
    xt = torch.tensor(x, device=dev)
    loss = torch.full((1,), 5.0, dtype=torch.float32, device=dev)
    y, g = torch.zeros(B, device=dev), torch.zeros(B, 6, device=dev)
    m.loss_grad(xt, torch.tensor(ty, device=dev), torch.tensor(tg, device=dev), cy, cg, loss)
    m.eval(xt, y, g)
    m.check()
    G = unpack(m.get_grad())
    yr, gr = omlp.input_grad(p, x.astype(np.float64), bf16=True)[:2]
    assert rel(y.cpu().numpy(), yr) < 4e-3 and rel(g.cpu().numpy(), gr) < 4e-3
    Lr = omlp.loss(p, x.astype(np.float64), ty, tg, cy, cg, bf16=True)
    assert abs(float(loss.item()) - Lr) < 8e-3 * abs(Lr)
    Gr = omlp.param_grad(p, x.astype(np.float64), ty, tg, cy, cg, bf16=True)
    for k in Gr:
        assert rel(G[k].reshape(-1), np.asarray(Gr[k]).reshape(-1)) < 2e-2, k
    m.close()


@pytest.mark.parametrize("n", [1, 31, 33, 100])
@pytest.mark.parametrize("degree", [0, 3, 4, 5, 6])
def test_surrogate_polynomial_degrees(n, degree):
    """Base law and polynomial part (FP64 on both sides, zero network) at the edges of the 32-point blocks."""
    import torch

    from paper_1908_08292_gb300.surrogate import MLP, SurrogateParams, surrogate_eval, work_floats
    F = synth.random_F(81, n, 3, 0.25)
    dev = torch.device("cuda:0")
    m = MLP(n)
    zero = {k: np.zeros_like(v) for k, v in net(82).items()}
    m.set_params(zero)
    sp = SurrogateParams(1.5, 0.9, 0.35, 0.02, 0.3)
    M = synth.random_field(83, 6, 6, 0.1)
    sp.set_Ca(M + M.T)
    c = 0.3 * synth.random_field(84, 1, 896, 1.0)[0]
    c[{0: 0, 3: 56, 4: 182, 5: 434, 6: 896}[degree]:] = 0.0
    sp.poly[:] = c.tolist()
    Ft = torch.tensor(F.reshape(n, 9), device=dev)
    P, A = torch.zeros(n, 9, dtype=torch.float64, device=dev), torch.zeros(n, 81, dtype=torch.float64, device=dev)
    P2, W = torch.zeros_like(P), torch.zeros(n, dtype=torch.float64, device=dev)
    ins = torch.zeros(n, dtype=torch.int32, device=dev)
    work = torch.zeros(work_floats(n), dtype=torch.float32, device=dev)
    surrogate_eval(m, sp, Ft, P, A, W, ins, work)
    surrogate_eval(m, sp, Ft, P2, None, None, ins, work)
    torch.cuda.synchronize()
    Wr, Pr, Ar = osur.evaluate(zero, F, 1.5, 0.9, 0.35, 0.02, Ca=M + M.T, poly=c)
    for got, ref in ((W[:, None], Wr[:, None]), (P, Pr.reshape(n, 9)), (P2, Pr.reshape(n, 9)), (A, Ar.reshape(n, 81))):
        err = np.linalg.norm(got.cpu().numpy() - ref, axis=1)
        assert np.all(err <= 1e-11 * np.maximum(np.linalg.norm(ref, axis=1), 1e-30))
    m.close()
