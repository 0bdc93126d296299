"""Elimination by levels against the lane-group form (which a call takes inside a
capture that finds no buffers): the same bits of log Z_R, d/dbeta and d/dJ, over
widths, several instances and tile edges, and a captured call's replay after a
larger call has grown the buffers."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


def _model(n, d, wu, insts, seed=11):
    gs, Ws, orders = [], [], []
    for k in range(insts):
        g = wl.random_regular(n + 8 * k, d, seed + n + d + k)
        W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, wu, restarts=1, seed=1)
        gs.append(g), Ws.append(W), orders.append(order)
    model = TNVAN(gs, Ws, [16], [0.7 + 0.2 * k for k in range(insts)], seed=3, elim_orders=orders)
    return gs, Ws, model


def _captured(fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        fn()
    return g


@pytest.mark.parametrize("n,d,wu,insts,batch", [
    (16, 3, 1, 1, 1), (64, 3, 1, 3, 33), (128, 3, 3, 1, 130), (90, 3, 4, 2, 31), (72, 4, 5, 1, 64), (60, 3, 7, 2, 300)])
def test_levels_equal_lane_groups(n, d, wu, insts, batch):
    gs, Ws, model = _model(n, d, wu, insts)
    D, m = sum(len(W) for W in Ws), sum(g.m for g in gs)
    spins = to_dev_spins(np.random.default_rng(n).choice([-1, 1], size=batch * D).astype(np.int8))
    model.ctx.reserve(batch)
    f64 = dict(dtype=torch.float64, device="cuda")
    out = [torch.full((insts * batch,), float("nan"), **f64) for _ in range(3)]
    dJ = torch.full((m,), float("nan"), **f64)
    logq = torch.zeros(insts * batch, dtype=torch.float32, device="cuda")
    grad = torch.empty_like(model.params)

    def run():
        model.ctx.contract(model.betas, batch, spins, tv.FP32, out[0])
        model.ctx.contract(model.betas, batch, spins, tv.FP32, out[1], out[2])
        model.ctx.backward(model.betas, batch, spins, out[0], logq, tv.FP32, grad, None, dJ)

    graph = _captured(run)
    graph.replay()
    torch.cuda.synchronize()
    lane = [t.clone() for t in (*out, dJ)]
    for t in (*out, dJ):
        t.fill_(float("nan"))
    run()
    torch.cuda.synchronize()
    for a, b in zip(lane, (*out, dJ)):
        assert torch.isfinite(b).all()
        if a is lane[3]:  # FP64 sums over the batch, in another order
            assert float((a - b).abs().max()) <= 1e-14 * max(1.0, float(b.abs().max()))
        else:
            assert torch.equal(a, b)


def test_captured_call_outlives_a_larger_one():
    _, Ws, model = _model(90, 3, 6, 1)
    D = len(Ws[0])
    s = to_dev_spins(np.random.default_rng(1).choice([-1, 1], size=9000 * D).astype(np.int8))
    lz = torch.empty(40, dtype=torch.float64, device="cuda")
    model.ctx.contract(model.betas, 40, s[:40 * D], tv.FP32, lz)
    torch.cuda.synchronize()
    ref = lz.clone()
    graph = _captured(lambda: model.ctx.contract(model.betas, 40, s[:40 * D], tv.FP32, lz))
    big = torch.empty(9000, dtype=torch.float64, device="cuda")
    db = torch.empty_like(big)
    model.ctx.contract(model.betas, 9000, s, tv.FP32, big, db)
    torch.cuda.synchronize()
    lz.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(lz, ref) and torch.equal(big[:40], ref)
