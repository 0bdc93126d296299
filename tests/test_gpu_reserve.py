"""tnvan_reserve: every call up to the reserved batch can be captured directly
after it (capture in global mode refuses allocations), elimination calls in the
form they take when called eagerly."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]

F64 = dict(dtype=torch.float64, device="cuda")


def _rrg(n, d, wu, hidden, insts=1):
    g = wl.random_regular(n, d, 77 + n + d)
    W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, wu, restarts=1, seed=1)
    return TNVAN([g] * insts, [W] * insts, hidden, [0.8] * insts, seed=3, elim_orders=[order] * insts)


def _lattice(Lx, Ly, cols, hidden, insts, dist="gauss"):
    gs = [wl.lattice(Lx, Ly, dist, 9 + k) for k in range(insts)]
    return TNVAN(gs, [wl.width_columns(Lx, Ly, cols)] * insts, hidden, [0.9] * insts, seed=3)


def _sk(n, rest, hidden, insts):
    return TNVAN([wl.sk(n, 3 + k) for k in range(insts)], [np.arange(n - rest, dtype=np.int32)] * insts, hidden,
                 [0.6] * insts, seed=3)


def _capture(fn, path=None):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph):
        fn()
    if path is not None:
        graph.debug_dump(str(path))
    graph.instantiate()
    return graph


CASES = {
    "levels": (lambda: _rrg(90, 3, 6, [64, 64]), 2000),
    "levels_global": (lambda: _rrg(500, 3, 8, [16], 2), 1500),
    "groups": (lambda: _rrg(300, 4, 10, [16]), 6000),
    "fused_one": (lambda: _lattice(16, 16, [4, 9, 14], [128, 128], 1), 20000),
    "fused": (lambda: _lattice(16, 16, [3, 7, 11, 15], [128, 128], 5), 16384),
    "strips": (lambda: _lattice(8, 8, [3], [16], 2), 3000),
    "wide": (lambda: _lattice(20, 10, [5, 12, 19], [32, 32], 2), 700),
    "chain": (lambda: _sk(64, 16, [256, 256], 3), 4096),
}


@pytest.mark.parametrize("name", CASES)
def test_capture_right_after_reserve(name):
    make, B = CASES[name]
    model = make()
    n = model.n
    D, m = sum(model.D), sum(model.n_edges)
    model.ctx.reserve(B)
    for b in (B, max(1, B - B // 3), 33):
        s = to_dev_spins(np.random.default_rng(b).choice([-1, 1], size=b * D).astype(np.int8))
        lz, db = torch.full((2, n * b), float("nan"), **F64)
        dJ = torch.full((m,), float("nan"), **F64)
        lz0 = torch.linspace(-1.0, 1.0, n * b, **F64)
        lq = torch.zeros(n * b, device="cuda")
        grads = {p: torch.full_like(model.params, float("nan")) for p in (tv.FP32, tv.TF32, tv.BF16)}
        outs = [lz, db, dJ, *grads.values()]

        def call():
            model.ctx.contract(model.betas, b, s, tv.FP32, lz)
            model.ctx.contract(model.betas, b, s, tv.FP32, lz, db)
            for p, g in grads.items():
                model.ctx.backward(model.betas, b, s, lz0, lq, p, g, None, dJ if p == tv.FP32 else None)

        graph = _capture(call)
        graph.replay()
        torch.cuda.synchronize()
        ref = [t.clone() for t in outs]
        for t in outs:
            t.fill_(float("nan"))
        call()
        torch.cuda.synchronize()
        for x, y in zip(ref, outs):
            assert torch.isfinite(y).all() and torch.equal(x, y)


def test_reserved_step_is_captured_by_levels(tmp_path):
    model = _rrg(128, 3, 5, [64, 64])
    B = 3000
    model.ctx.reserve(B)
    out = model.buffers(B)
    grad, m, v = (torch.zeros_like(model.params) for _ in range(3))
    db, dJ = torch.empty(B, **F64), torch.empty(sum(model.n_edges), **F64)
    path = tmp_path / "g.dot"
    _capture(lambda: model.ctx.train_step(model.betas, B, 3, 0, tv.BF16, *out, db, dJ, grad, m, v, 0.01, 0.9, 0.999,
                                          1e-8, 1), path).replay()
    torch.cuda.synchronize()
    text = path.read_text()
    assert "general_levels_kernel" in text and "general_levels_dJ_kernel" in text and "14general_kernel" not in text
    assert torch.isfinite(model.params).all() and torch.isfinite(dJ).all()
