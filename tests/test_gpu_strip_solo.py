"""Lattice contraction by pairs of (strip, 32 samples) and by one thread a sample
through all strips: short strips over many samples take the latter, and a
sample's bits do not depend on it."""
import numpy as np
import pytest
import torch

from oracle import transfer
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]


def _solo(fn, path):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        fn()
    graph.debug_dump(str(path))
    text = path.read_text()
    assert "13strips_kernelI" in text
    return any(f"13strips_kernelILb{db}ELi{w}ELb1E" in text for db in (0, 1) for w in (3, 4))


# (Lx, Ly, columns of W, instances, large batch, solo there): widths 1 to 4, W at an edge,
# no strip at all, 128 states (8 x 8), more than 128 (12 x 12), and a full last tile or one sample of it
CASES = [(4, 4, (3,), 5, 8192, True), (5, 5, (2, 4), 2, 30_001, True), (7, 4, (3, 5), 1, 39_001, True),
         (9, 9, (1, 3, 5, 7), 5, 8193, True), (3, 5, (0, 1, 2), 1, 40_000, True), (8, 8, (3, 7), 5, 9_999, True),
         (2, 12, (0,), 1, 38_912, False), (12, 12, (4, 9), 5, 9_999, False)]


@pytest.mark.parametrize("Lx,Ly,cols,insts,large,solo", CASES)
@pytest.mark.parametrize("db", [False, True], ids=["lz", "dbeta"])
def test_same_bits(Lx, Ly, cols, insts, large, solo, db, tmp_path):
    small = 203
    W = wl.width_columns(Lx, Ly, list(cols))
    graphs = [wl.lattice(Lx, Ly, "gauss", k + 1) for k in range(insts)]
    model = TNVAN(graphs, [W] * insts, [8], list(np.linspace(0.4, 1.2, insts)), seed=2)
    D, rng = len(W), np.random.default_rng(5)
    spins = rng.choice([-1, 1], size=(insts, large, D)).astype(np.int8)

    def run(b):
        s = torch.as_tensor(np.ascontiguousarray(spins[:, :b])).cuda().reshape(-1)
        lz = torch.full((insts * b,), 7.0, dtype=torch.float64, device="cuda")
        d = torch.full_like(lz, 7.0) if db else None

        def call():
            model.ctx.contract(model.betas, b, s, tv.FP32, lz, d)

        call()
        torch.cuda.synchronize()
        out = [lz.view(insts, b)[:, :small].clone()] + ([d.view(insts, b)[:, :small].clone()] if db else [])
        assert not (lz == 7.0).any()
        return _solo(call, tmp_path / f"{b}.dot"), out

    by_pairs, a = run(small)
    by_solo, b = run(large)
    assert (by_pairs, by_solo) == (False, solo)
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    for k in (0, insts - 1):
        g = graphs[k]
        ref = transfer.log_zr_lattice(g.n, g.ei, g.ej, g.J, float(model.betas[k]), W,
                                      torch.as_tensor(spins[k, :16].astype(np.float64)), g.Lx)
        assert (b[0][k, :16].cpu() - ref).abs().max().item() / g.n < 1e-6
