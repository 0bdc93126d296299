"""Graphs without bonds: log Z_R = (n - n_w) ln 2, zero derivatives, and the
adjoint call accepted beside a graph with bonds and alone."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beside", [False, True])
def test_no_bonds(beside):
    n, nw, batch = 24, 3, 40
    none = np.zeros(0, np.int32)
    g = wl.Graph(n, none, none, np.zeros(0))
    gs = [g] + ([wl.random_regular(24, 3, 5)] if beside else [])
    model = TNVAN(gs, [np.arange(nw, dtype=np.int32)] * len(gs), [8], [0.7] * len(gs), seed=1)
    assert model.ctx.instance_info(0)["kind"] == 2
    k = len(gs)
    s = to_dev_spins(np.random.default_rng(0).choice([-1, 1], size=k * batch * nw).astype(np.int8))
    lz, db = torch.empty(2, k * batch, dtype=torch.float64, device="cuda")
    dJ = torch.full((1 + sum(h.m for h in gs),), 7.0, dtype=torch.float64, device="cuda")
    model.ctx.contract(model.betas, batch, s, tv.FP32, lz, db)
    model.ctx.backward(model.betas, batch, s, lz, torch.zeros(k * batch, device="cuda"), tv.FP32,
                       torch.empty_like(model.params), db, dJ)
    torch.cuda.synchronize()
    # FP32 sums of powers of two
    assert torch.allclose(lz[:batch].cpu(), torch.full((batch,), (n - nw) * np.log(2.0), dtype=torch.float64), rtol=1e-6)
    assert (db[:batch] == 0).all()
    assert float(dJ[-1]) == 7.0 and torch.isfinite(dJ).all()
