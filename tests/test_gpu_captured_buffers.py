"""A captured call keeps its workspaces when later, larger calls grow the
context's buffers: replayed afterwards it gives the same bits."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu

F64 = dict(dtype=torch.float64, device="cuda")


def _replay_after(small, outs, large):
    """Runs `small`, captures it, runs `large`, replays; outs: its output tensors."""
    small()
    torch.cuda.synchronize()
    ref = [t.clone() for t in outs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        small()
    large()
    torch.cuda.synchronize()
    # what the larger call freed is handed out again
    fill = [torch.full((1 << 22,), float("nan"), device="cuda") for _ in range(8)]
    for t in outs:
        t.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.isnan(f).all() for f in fill)
    for a, b in zip(ref, outs):
        assert torch.isfinite(b).all() and torch.equal(a, b)


@pytest.mark.parametrize("precision", [tv.FP32, tv.TF32, tv.BF16])
@pytest.mark.parametrize("kind", ["elimination", "strips"])
def test_backward_outlives_growth(kind, precision):
    if kind == "elimination":
        g = wl.random_regular(90, 3, 101)
        W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, 6, restarts=1, seed=1)
        model = TNVAN([g], [W], [256, 256], [0.8], seed=3, elim_orders=[order])
    else:
        g = wl.lattice(8, 8, "gauss", 5)
        W = wl.width_columns(8, 8, [3])
        model = TNVAN([g], [W], [256, 256], [0.8], seed=3)
    D, big = len(W), 9000
    s = to_dev_spins(np.random.default_rng(1).choice([-1, 1], size=big * D).astype(np.int8))
    grad = torch.empty_like(model.params)

    def call(b):
        lz = torch.linspace(-1.0, 1.0, b, **F64)
        lq = torch.zeros(b, device="cuda")
        db, dJ = torch.empty(b, **F64), torch.empty(g.m, **F64)
        return (lambda: model.ctx.backward(model.betas, b, s[:b * D], lz, lq, precision, grad, db, dJ)), (grad, db, dJ)

    small, outs = call(40)
    large, _ = call(big)
    _replay_after(small, outs, large)


def test_wide_strips_outlive_growth():
    g = wl.lattice(16, 8, "pm1", 5)
    W = wl.width_columns(16, 8, [8])
    model = TNVAN([g], [W], [16], [0.7], seed=3)
    D, big = len(W), 9000
    s = to_dev_spins(np.random.default_rng(2).choice([-1, 1], size=big * D).astype(np.int8))
    lz, lzb = torch.empty(40, **F64), torch.empty(big, **F64)
    _replay_after(lambda: model.ctx.contract(model.betas, 40, s[:40 * D], tv.FP32, lz), (lz,),
                  lambda: model.ctx.contract(model.betas, big, s, tv.FP32, lzb))
