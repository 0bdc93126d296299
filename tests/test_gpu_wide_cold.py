"""Wide strips at low temperature: frustrated rows whose largest entry is far
below 1 keep the precision of FP32 in log Z_R."""
import numpy as np
import pytest
import torch

from oracle import general
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,col,dist,beta", [
    (25, 10, 12, "pm1", 5.0), (25, 10, 12, "gauss", 5.0), (16, 14, 8, "pm1", 7.0), (21, 12, 10, "gauss", 7.0),
    (11, 12, 5, "gauss", 15.0), (6, 6, 5, "gauss", 20.0)])
def test_cold_frustrated_strips(Lx, Ly, col, dist, beta):
    g = wl.lattice(Lx, Ly, dist, 3)
    W = wl.width_columns(Lx, Ly, [col])
    batch = 200
    s = np.random.default_rng(1).choice([-1, 1], size=(batch, len(W))).astype(np.int8)
    model = TNVAN([g], [W], [8], [beta], seed=1)
    lz = torch.empty(batch, dtype=torch.float64, device="cuda")
    model.ctx.profile(True)
    model.ctx.contract(model.betas, batch, to_dev_spins(s), tv.FP32, lz)
    torch.cuda.synchronize()
    assert "wide_strips" in model.ctx.profile_read()
    ref = general.log_zr_general(g.n, g.ei, g.ej, g.J, beta, W, torch.as_tensor(s.astype(np.float64)),
                                 enum_max=0).numpy()
    # the parity bound of the FP32 contractions, per spin
    assert np.abs(lz.cpu().numpy() - ref).max() / g.n <= 1e-6
