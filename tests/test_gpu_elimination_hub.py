"""Eliminating a spin that many tables contain (the hub of a star whose leaves
go first): log Z_R, d/dbeta and d/dJ against the star's closed form, below and
above 255 tables."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaves", [3, 255, 256, 300])
def test_star(leaves):
    """Hub 0, leaves 1..n, 15 width-set spins with every 15th leaf each (too many for component tables); all
    bonds 1, beta 1, at most two width-set spins down, so that the hub's product stays inside FP32's range."""
    nw, beta, batch = 15, 1.0, 70
    lf = np.arange(1, leaves + 1, dtype=np.int32)
    wi = (lf - 1) % nw
    ei = np.concatenate([np.zeros(leaves, np.int32), lf])
    ej = np.concatenate([lf, leaves + 1 + wi]).astype(np.int32)
    g = wl.Graph(1 + leaves + nw, ei, ej, np.ones(2 * leaves))
    W = np.arange(leaves + 1, leaves + 1 + nw, dtype=np.int32)
    order = np.concatenate([lf, [0]]).astype(np.int32)
    model = TNVAN([g], [W], [16], [beta], seed=1, elim_orders=[order])
    rng = np.random.default_rng(leaves)
    s = np.ones((batch, nw))
    for b in range(1, batch):
        s[b, rng.choice(nw, size=1 + b % 2, replace=False)] = -1.0
    h = s[:, wi]  # [batch, leaves] the leaves' fields
    a = np.stack([1.0 + h, -1.0 + h])  # [hub state, batch, leaves]
    f = np.log(2.0 * np.cosh(beta * a)).sum(2)
    lz = np.logaddexp(f[0], f[1])
    p = np.exp(f - lz)
    t = np.tanh(beta * a)
    db = (p * (a * t).sum(2)).sum(0)
    dJ_hub = beta * (p[0][:, None] * t[0] - p[1][:, None] * t[1]).mean(0)
    dJ_leaf = beta * (h * (p[0][:, None] * t[0] + p[1][:, None] * t[1])).mean(0)

    dev = to_dev_spins(s)
    out = torch.full((3, batch), float("nan"), dtype=torch.float64, device="cuda")
    dJ = torch.full((g.m,), float("nan"), dtype=torch.float64, device="cuda")
    model.ctx.contract(model.betas, batch, dev, tv.FP32, out[0])
    model.ctx.contract(model.betas, batch, dev, tv.FP32, out[1], out[2])
    model.ctx.backward(model.betas, batch, dev, out[0].clone(), torch.zeros(batch, device="cuda"), tv.FP32,
                       torch.empty_like(model.params), None, dJ)
    torch.cuda.synchronize()
    out, dJ = out.cpu().numpy(), dJ.cpu().numpy()
    # FP32 products of `leaves` tables: a few roundings of 6e-8 per table and spin
    tol = 1e-6 * g.n
    assert np.abs(out[0] - lz).max() <= tol and np.abs(out[1] - lz).max() <= tol
    assert np.abs(out[2] - db).max() <= 2 * tol  # |a| <= 2
    assert np.abs(dJ - np.concatenate([dJ_hub, dJ_leaf])).max() <= 2e-5
