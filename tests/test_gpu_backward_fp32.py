"""The FP32 backward of Eq. 10 at the edges of its tiles (32 samples, 128
units, 32 inputs a stage, 64 x 64 gradient blocks) against the oracle's
REINFORCE gradient: no, one and two hidden layers, widths that are not
multiples of four, one spin, ragged batches."""
import numpy as np
import pytest
import torch

from oracle import estimators as est
from oracle import made
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,hidden,batch", [
    (1, [], 33), (7, [], 33), (1, [5], 32), (4, [16], 100), (37, [130], 31), (5, [3, 2], 65), (33, [35, 129], 64),
    (64, [128, 128], 700), (70, [257, 66], 97), (130, [64, 300], 40)])
def test_fp32_backward_matches_oracle(D, hidden, batch):
    from paper_2504_12037_gb300.model import TNVAN

    # two different instances side by side: W = the first D spins
    graphs = [wl.sk(D + 4, 5), wl.sk(D + 4, 6)]
    Ws = [np.arange(D, dtype=np.int32)] * 2
    model = TNVAN(graphs, Ws, hidden, [0.7, 1.2], seed=11, init_scale=1.5)
    rng = np.random.default_rng(D)
    s = rng.choice([-1.0, 1.0], size=(2, batch, D))
    lz = rng.normal(-50.0, 3.0, size=(2, batch))
    lq = rng.normal(-0.7 * D, 1.0, size=(2, batch)).astype(np.float32)
    grad = torch.full_like(model.params, float("nan"))
    model.ctx.backward(model.betas, batch, to_dev_spins(s), torch.as_tensor(lz.reshape(-1)).cuda(),
                       torch.as_tensor(lq.reshape(-1)).cuda(), tv.FP32, grad)
    torch.cuda.synchronize()
    for k in range(2):
        p = model.params[model.offsets[k]:model.offsets[k + 1]].cpu().numpy().astype(np.float64)
        w = est.reinforce_weights(torch.as_tensor(lz[k]), torch.as_tensor(lq[k].astype(np.float64)), model.betas[k])
        ref = est.surrogate_grad(p, D, hidden, torch.as_tensor(s[k]), w)
        g = grad[model.offsets[k]:model.offsets[k + 1]].cpu().double()
        assert torch.isfinite(g).all()
        # FP32 sums of a few hundred terms of the gradient's own size
        assert float((g - ref).abs().max()) <= 2e-5 * float(ref.abs().max())
