"""Batch sizes at the edges of the tiles of the FP32 sampler, the F_q reduction
and the strip contraction."""
import numpy as np
import pytest
import torch

from oracle import made
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl

from gpu_helpers import check_sample_agreement, oracle_samples, to_dev_spins

pytestmark = pytest.mark.gpu

TOL_FP32 = 1e-6


@pytest.mark.parametrize("D,hidden,batch", [
    (1, [], 9), (5, [], 7), (6, [40], 8), (20, [16], 193), (33, [35, 17], 65), (12, [256, 256], 31), (64, [128, 128], 500)])
def test_fp32_sampler_tiles(D, hidden, batch):
    from paper_2504_12037_gb300.model import TNVAN

    graphs = [wl.sk(D + 3, 1), wl.sk(D + 3, 2)]
    model = TNVAN(graphs, [np.arange(D, dtype=np.int32)] * 2, hidden, [0.5, 1.0], seed=4, init_scale=2.0)
    spins, logq, _ = model.sample(batch, 21, 3, tv.FP32)
    torch.cuda.synchronize()
    for k in range(2):
        p = model.params[model.offsets[k]:model.offsets[k + 1]].cpu().numpy()
        s_or, p_or, u = oracle_samples(p, D, hidden, 21, 3, k, batch)
        s_gpu = model.spins_of(spins, k, batch).cpu().numpy().astype(np.float64)
        same = check_sample_agreement(s_gpu, s_or.numpy(), u, p_or.numpy())
        lq = made.log_q(torch.as_tensor(p, dtype=torch.float64), D, hidden, s_or)
        err = (logq[k * batch:(k + 1) * batch].cpu().double() - lq).abs()[torch.as_tensor(same)]
        assert float(err.max()) / graphs[k].n <= TOL_FP32


@pytest.mark.parametrize("batch", [1, 2, 63, 64, 65, 129, 2048, 2049, 4097, 20001])
@pytest.mark.parametrize("bad", [False, True])
def test_reduction_chunks(batch, bad):
    from paper_2504_12037_gb300.model import TNVAN

    g = wl.lattice(4, 4, "gauss", 3)
    model = TNVAN([g] * 3, [wl.width_columns(4, 4, [1])] * 3, [8], [0.3, 0.7, 1.1], seed=1)
    rng = np.random.default_rng(batch)
    lz = rng.normal(0.0, 40.0, size=(3, batch)) + np.array([[-900.0], [0.0], [2500.0]])
    lq = rng.normal(-30.0, 2.0, size=(3, batch)).astype(np.float32)
    if bad:
        lz[0, 0] = np.inf
        lz[1, batch // 2] = np.nan
        lq[2, :] = np.nan  # no finite value at all
    out = torch.empty(24, dtype=torch.float64, device="cuda")
    model.ctx.reduce(model.betas, batch, torch.as_tensor(lz.reshape(-1)).cuda(), torch.as_tensor(lq.reshape(-1)).cuda(),
                     out)
    torch.cuda.synchronize()
    out = out.view(3, 8).cpu().numpy()
    for k in range(3):
        l = lz[k] - lq[k].astype(np.float64)
        fin = l[np.isfinite(l)]
        n = len(fin)
        assert out[k, 5] == batch - n and out[k, 7] == n
        if n == 0:
            assert np.isnan(out[k, [0, 1, 3, 4]]).all()
            continue
        m = fin.max()
        lzis = m + np.log(np.exp(fin - m).sum()) - np.log(n)
        var = fin.var(ddof=1) if n > 1 else 0.0
        b = model.betas[k]
        ref = np.array([-fin.mean() / b, -lzis / b, np.sqrt(var) / (b * np.sqrt(n)), lzis, fin.mean()])
        # float-float moment sums (48 bits) of values up to a few thousand
        assert np.abs(out[k, :5] - ref).max() <= 1e-9 * max(1.0, np.abs(fin).max())
        assert abs(out[k, 6] - var) <= 1e-9 * max(1.0, var)


@pytest.mark.parametrize("L,cols", [(4, [1]), (9, [4]), (12, [3, 7, 11])])
def test_strip_contraction_tiles_agree(L, cols):
    # the same configurations in calls of one sample, a ragged tile, and enough
    # samples for two tiles a CTA: the same bits
    from paper_2504_12037_gb300.model import TNVAN

    g = wl.lattice(L, L, "gauss", 5)
    W = wl.width_columns(L, L, cols)
    model = TNVAN([g], [W], [8], [0.9], seed=2)
    big = 400_000
    s = np.random.default_rng(3).choice([-1, 1], size=(big, len(W))).astype(np.int8)
    d = to_dev_spins(s)

    def run(n, db):
        lz = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        dl = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") if db else None
        model.ctx.contract(model.betas, n, d[:n * len(W)].clone(), tv.FP32, lz, dl)
        torch.cuda.synchronize()
        return lz.cpu(), dl.cpu() if db else None

    lz0, _ = run(big, False)
    lz1, db1 = run(big, True)
    assert torch.equal(lz0, lz1) and torch.isfinite(db1).all()
    for n in (1, 33, 130):
        lz, db = run(n, True)
        assert torch.equal(lz, lz1[:n]) and torch.equal(db, db1[:n])
        assert torch.equal(run(n, False)[0], lz)
