"""Log-weights far from zero (large beta or many spins): log Z_IS and F_IS against
NumPy over the whole range of FP64, with all chunks or only some of them far out."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 65, 700, 5000])
@pytest.mark.parametrize("off", [5e8, 6.5e8, 8e8, 1e9, -1e9, -6.5e8, 3e12, -3e12, 1e40, -1e40])
@pytest.mark.parametrize("part", [False, True])
def test_far_log_weights(batch, off, part):
    from paper_2504_12037_gb300.model import TNVAN

    g = wl.lattice(4, 4, "gauss", 3)
    model = TNVAN([g] * 2, [wl.width_columns(4, 4, [1])] * 2, [8], [0.5, 1.25], seed=1)
    rng = np.random.default_rng(batch)
    lz = rng.normal(0.0, 20.0, size=(2, batch))
    far = np.arange(batch) % 128 < 64 if part else np.ones(batch, bool)
    lz[:, far] = off * (1.0 + 1e-9 * rng.normal(size=(2, far.sum())))
    lq = rng.normal(-30.0, 2.0, size=(2, batch)).astype(np.float32)
    if batch > 1:
        lz[1, batch - 1] = np.inf
    out = torch.empty(16, dtype=torch.float64, device="cuda")
    model.ctx.reduce(model.betas, batch, torch.as_tensor(lz.reshape(-1)).cuda(), torch.as_tensor(lq.reshape(-1)).cuda(),
                     out)
    torch.cuda.synchronize()
    out = out.view(2, 8).cpu().numpy()
    for k in range(2):
        l = lz[k] - lq[k].astype(np.float64)
        fin = l[np.isfinite(l)]
        n, m, b = len(fin), fin.max(), model.betas[k]
        ref = m + np.log(np.exp(fin - m).sum()) - np.log(n)
        assert out[k, 5] == batch - n and out[k, 7] == n
        # the largest l, a scale and their difference each within half a unit in the last place
        tol = 4 * 2.0 ** -52 * abs(m) + 1e-11
        assert abs(out[k, 3] - ref) <= tol
        assert abs(out[k, 1] + ref / b) <= 2 * tol / b
        if abs(off) < 1e18:  # the FP32 pairs of the moment sums hold squares up to 3e38
            # 48-bit sums
            assert abs(out[k, 4] - fin.mean()) <= 1e-9 * np.abs(fin).max()
