"""The lane = sample elimination kernels: the same bits as the lane-group form
that longer calls take, and d/dJ against the oracle, over table sizes (widths),
tile edges and several instances."""
import numpy as np
import pytest
import torch

from oracle import general
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


def _model(n, d, wu, insts=1):
    g = wl.random_regular(n, d, 77 + n + d)
    W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, wu, restarts=1, seed=1)
    return g, W, TNVAN([g] * insts, [W] * insts, [16], [0.8] * insts, seed=3, elim_orders=[order] * insts)


@pytest.mark.parametrize("n,d,wu,db", [(500, 3, 8, True), (500, 3, 8, False), (500, 3, 5, False), (240, 4, 8, True)])
def test_small_and_large_calls_agree(n, d, wu, db):
    g, W, model = _model(n, d, wu)
    big = 12000
    s = np.random.default_rng(5).choice([-1, 1], size=(big, len(W))).astype(np.int8)
    dev = to_dev_spins(s.reshape(-1))

    def run(b):
        lz = torch.full((b,), float("nan"), dtype=torch.float64, device="cuda")
        dl = torch.full((b,), float("nan"), dtype=torch.float64, device="cuda") if db else None
        model.ctx.contract(model.betas, b, dev[:b * len(W)].clone(), tv.FP32, lz, dl)
        torch.cuda.synchronize()
        return lz.cpu(), dl.cpu() if db else lz.cpu()

    lz0, dl0 = run(big)
    assert torch.isfinite(lz0).all() and torch.isfinite(dl0).all()
    for b in (1, 31, 33, 1000):
        lz, dl = run(b)
        assert torch.equal(lz, lz0[:b]) and torch.equal(dl, dl0[:b])


@pytest.mark.parametrize("n,d,wu,batch,insts", [(64, 3, 1, 3, 1), (90, 3, 4, 33, 2), (120, 3, 6, 31, 1), (80, 4, 7, 65, 3),
                                                (120, 4, 9, 5, 1)])
def test_dJ_matches_oracle(n, d, wu, batch, insts):
    g, W, model = _model(n, d, wu, insts)
    rng = np.random.default_rng(n)
    s = rng.choice([-1, 1], size=(insts, batch, len(W))).astype(np.int8)
    dev = to_dev_spins(s.reshape(-1))
    lz = torch.empty(insts * batch, dtype=torch.float64, device="cuda")
    model.ctx.contract(model.betas, batch, dev, tv.FP32, lz)
    dJ = torch.empty(insts * g.m, dtype=torch.float64, device="cuda")
    grad = torch.empty_like(model.params)
    model.ctx.backward(model.betas, batch, dev, lz, torch.zeros(insts * batch, dtype=torch.float32, device="cuda"),
                       tv.FP32, grad, None, dJ)
    torch.cuda.synchronize()
    for k in range(insts):
        Jt = torch.tensor(g.J, dtype=torch.float64, requires_grad=True)
        ref = general.log_zr_general(g.n, g.ei, g.ej, Jt, 0.8, W, torch.as_tensor(s[k], dtype=torch.float64))
        (rj,) = torch.autograd.grad(ref.mean(), Jt)
        assert float((lz[k * batch:(k + 1) * batch].cpu() - ref.detach()).abs().max()) / g.n <= 1e-6
        # FP32 sums, as in the planned graphs' adjoint test
        assert float((dJ[k * g.m:(k + 1) * g.m].cpu() - rj).abs().max()) <= 2e-5 * max(1.0, float(rj.abs().max()))
