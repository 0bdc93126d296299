"""The wide-strip contraction's change of layout from row to row: strips of 9
to 12 columns with one row, an even and an odd number of rows and more than
32, W neighbours on both sides, one side or the other, against the FP64
oracle."""
import numpy as np
import pytest
import torch

from oracle import transfer
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,L,side,dist", [
    (9, 5, "both", "gauss"), (10, 1, "both", "gauss"), (10, 2, "left", "pm1"), (10, 33, "right", "gauss"),
    (11, 3, "both", "pm1"), (11, 34, "left", "gauss"), (12, 2, "right", "ferro"), (12, 33, "both", "gauss")])
def test_wide_strip_rows(w, L, side, dist):
    from paper_2504_12037_gb300.model import TNVAN

    cols = {"both": [0, w + 1], "left": [0], "right": [w]}[side]
    Lx = w + len(cols)
    g = wl.lattice(Lx, L, dist, seed=w + L)
    W = wl.width_columns(Lx, L, cols)
    order = np.asarray([v for v in range(g.n) if v not in set(W.tolist())], np.int32)
    model = TNVAN([g], [W], [16], [0.7], seed=3, elim_orders=[order])
    B = 9
    s = np.random.default_rng(w * L).choice([-1.0, 1.0], size=(B, len(W)))
    lz = torch.empty(B, dtype=torch.float64, device="cuda")
    model.ctx.contract(model.betas, B, to_dev_spins(s), tv.FP32, lz)
    torch.cuda.synchronize()
    ref = transfer.log_zr_lattice(g.n, g.ei, g.ej, g.J, 0.7, W, torch.as_tensor(s), Lx)
    assert float((lz.cpu() - ref).abs().max()) / g.n <= 1e-6
