"""Which form an elimination call takes (by levels or in lane groups), read off
the kernels a capture records, and that both forms give the same bits, also where
the level form keeps its tables in global memory."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]


def _recorded(fn, path):
    """Names (mangled) of the kernels `fn` launches, from a capture's graph."""
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        fn()
    graph.debug_dump(str(path))
    return path.read_text()


def _form(text):
    levels, groups = "general_levels_kernel" in text, "14general_kernel" in text
    assert levels != groups
    return "levels" if levels else "groups"


# tables and derivatives of two levels in global memory; tables in shared memory, derivatives in global;
# both in shared memory with four lanes a sample; tables only, four lanes a sample; two lanes a sample
@pytest.mark.parametrize("n,d,wu,db,small,large", [
    (1000, 3, 10, True, 4800, 4896), (500, 3, 8, True, 4864, 4865), (500, 3, 4, True, 19456, 32768),
    (1000, 3, 4, True, 19456, 32768), (1000, 3, 4, False, 4096, 32768),
    (1000, 3, 2, True, 4096, 65536), (1000, 3, 2, False, 4096, 65536)])
def test_forms_agree(n, d, wu, db, small, large, tmp_path):
    g = wl.random_regular(n, d, 77 + n + d)
    W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, wu, restarts=1, seed=1)
    model = TNVAN([g], [W], [16], [0.8], seed=3, elim_orders=[order])
    s = to_dev_spins(np.random.default_rng(5).choice([-1, 1], size=large * len(W)).astype(np.int8))

    def run(b):
        lz = torch.full((b,), float("nan"), dtype=torch.float64, device="cuda")
        dl = torch.full((b,), float("nan"), dtype=torch.float64, device="cuda") if db else None

        def call():
            model.ctx.contract(model.betas, b, s[:b * len(W)], tv.FP32, lz, dl)

        call()
        torch.cuda.synchronize()
        out = (lz.clone(), dl.clone() if db else lz.clone())
        return out, _form(_recorded(call, tmp_path / f"{b}.dot"))

    (lz0, dl0), form0 = run(small)
    (lz1, dl1), form1 = run(large)
    assert (form0, form1) == ("levels", "groups")
    assert torch.isfinite(lz1).all() and torch.isfinite(dl1).all()
    assert torch.equal(lz0, lz1[:small]) and torch.equal(dl0, dl1[:small])


@pytest.mark.parametrize("db", [False, True])
def test_ladder_forms_agree(db, tmp_path):
    """Few tasks a level: lane groups over many samples, tables in shared memory."""
    n, w = 50, 5
    ij = [(v, v + w) for v in range(n - w)] + [(v, v + 1) for v in range(n - 1) if (v + 1) % w]
    ei, ej = (np.asarray(x, np.int32) for x in zip(*ij))
    g = wl.Graph(n, ei, ej, np.random.default_rng(1).normal(size=len(ij)))
    W = np.random.default_rng(7).choice(n, 14, replace=False).astype(np.int32)
    model = TNVAN([g], [W], [8], [0.8], seed=1)
    small, large = 8000, 65536
    s = to_dev_spins(np.random.default_rng(2).choice([-1, 1], size=large * len(W)).astype(np.int8))
    got = []
    for b in (small, large):
        lz, dl = torch.full((2, b), float("nan"), dtype=torch.float64, device="cuda")

        def call():
            model.ctx.contract(model.betas, b, s[:b * len(W)], tv.FP32, lz, dl if db else None)

        call()
        torch.cuda.synchronize()
        got.append((_form(_recorded(call, tmp_path / f"{b}.dot")), lz, dl if db else lz))
    assert [f for f, _, _ in got] == ["levels", "groups"]
    for a, c in zip(got[0][1:], got[1][1:]):
        assert torch.isfinite(c).all() and torch.equal(a, c[:small])


@pytest.mark.parametrize("n,d,wu,insts,batch", [
    (64, 3, 1, 3, 33), (128, 3, 3, 1, 130), (90, 3, 4, 2, 65), (60, 3, 7, 2, 300), (500, 3, 8, 1, 200)])
def test_adjoint_forms_agree(n, d, wu, insts, batch, tmp_path):
    """A capture that finds no buffers records lane groups; log Z_R and d/dbeta have the same bits, d/dJ is
    added up over the batch in FP64 in another order."""
    gs = [wl.random_regular(n + 8 * k, d, 11 + n + d + k) for k in range(insts)]
    plans = [tv.find_width_set(g.n, g.ei, g.ej, wu, restarts=1, seed=1)[:2] for g in gs]
    model = TNVAN(gs, [W for W, _ in plans], [16], [0.7 + 0.2 * k for k in range(insts)], seed=3,
                  elim_orders=[o for _, o in plans])
    D, m = sum(model.D), sum(model.n_edges)
    s = to_dev_spins(np.random.default_rng(n).choice([-1, 1], size=batch * D).astype(np.int8))
    model.ctx.reserve(1)
    lz, lz1, db = torch.full((3, insts * batch), float("nan"), dtype=torch.float64, device="cuda")
    dJ = torch.full((m,), float("nan"), dtype=torch.float64, device="cuda")
    lq, grad = torch.zeros(insts * batch, device="cuda"), torch.empty_like(model.params)

    def call():
        model.ctx.contract(model.betas, batch, s, tv.FP32, lz)
        model.ctx.contract(model.betas, batch, s, tv.FP32, lz1, db)
        model.ctx.backward(model.betas, batch, s, lz, lq, tv.FP32, grad, None, dJ)

    def run(path):
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        graph.enable_debug_mode()
        with torch.cuda.graph(graph, capture_error_mode="relaxed"):
            call()
        graph.debug_dump(str(path))
        graph.instantiate()
        graph.replay()
        torch.cuda.synchronize()
        text = path.read_text()
        return _form(text), "general_levels_dJ_kernel" in text, [t.clone() for t in (lz, lz1, db, dJ)]

    form0, dj0, out0 = run(tmp_path / "groups.dot")
    call()  # allocates
    form1, dj1, out1 = run(tmp_path / "levels.dot")
    assert (form0, dj0, form1, dj1) == ("groups", False, "levels", True)
    for a, b in zip(out0[:3], out1[:3]):
        assert torch.isfinite(b).all() and torch.equal(a, b)
    assert float((out0[3] - out1[3]).abs().max()) <= 1e-14 * max(1.0, float(out1[3].abs().max()))


def test_large_untabulated_call_stays_by_levels(tmp_path):
    """Lane groups keep the tables in shared memory: few CTAs an SM, slower at any batch."""
    g = wl.random_regular(500, 3, 77 + 503)
    W, order, _, _ = tv.find_width_set(g.n, g.ei, g.ej, 4, restarts=1, seed=1)
    model = TNVAN([g], [W], [16], [0.8], seed=3, elim_orders=[order])
    b = 20000
    s = to_dev_spins(np.random.default_rng(5).choice([-1, 1], size=b * len(W)).astype(np.int8))
    lz, dl = torch.empty(2, b, dtype=torch.float64, device="cuda")

    def call():
        model.ctx.contract(model.betas, b, s, tv.FP32, lz, dl)

    call()
    assert _form(_recorded(call, tmp_path / "g.dot")) == "levels"
