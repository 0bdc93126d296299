"""The BF16 backward chain and its weight gradients at the edges of their tiles
(128 samples, 16-unit padding, 32-input weight stages, 128-row gradient
blocks), against the oracle's REINFORCE gradient with the reduced-precision
bounds: no, one and two hidden layers, widths that are not multiples of 8, up
to the 256 limit, ragged batches, instances of different sizes in one call."""
import numpy as np
import pytest
import torch

from oracle import estimators as est
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ds,hidden,batch", [
    ((7, 20), [], 129), ((4, 33), [16], 100), ((37, 5), [130], 257), ((33, 16), [35, 129], 64),
    ((97, 48), [256, 256], 300), ((256, 3), [128, 200], 130), ((17, 130), [250, 24], 128)])
def test_bf16_chain_matches_oracle(Ds, hidden, batch):
    from paper_2504_12037_gb300.model import TNVAN

    graphs = [wl.sk(D + 4, 5 + D) for D in Ds]
    Ws = [np.arange(D, dtype=np.int32) for D in Ds]
    model = TNVAN(graphs, Ws, hidden, [0.7, 1.2], seed=11, init_scale=1.5)
    rng = np.random.default_rng(Ds[0])
    s = [rng.choice([-1.0, 1.0], size=(batch, D)) for D in Ds]
    lz = rng.normal(-50.0, 3.0, size=(2, batch))
    lq = rng.normal(-20.0, 1.0, size=(2, batch)).astype(np.float32)
    grad = torch.full_like(model.params, float("nan"))
    model.ctx.profile(True)
    model.ctx.backward(model.betas, batch, to_dev_spins(np.concatenate([x.reshape(-1) for x in s])),
                       torch.as_tensor(lz.reshape(-1)).cuda(), torch.as_tensor(lq.reshape(-1)).cuda(), tv.BF16, grad)
    torch.cuda.synchronize()
    assert "bwd_chain" in model.ctx.profile_read()
    for k, D in enumerate(Ds):
        p = model.params[model.offsets[k]:model.offsets[k + 1]].cpu().numpy().astype(np.float64)
        w = est.reinforce_weights(torch.as_tensor(lz[k]), torch.as_tensor(lq[k].astype(np.float64)), model.betas[k])
        ref = est.surrogate_grad(p, D, hidden, torch.as_tensor(s[k]), w)
        g = grad[model.offsets[k]:model.offsets[k + 1]].cpu().double()
        assert torch.isfinite(g).all()
        fro = float((g - ref).norm() / ref.norm())
        cos = float(torch.nn.functional.cosine_similarity(g, ref, dim=0))
        assert fro <= 1e-1 and cos >= 0.99, (k, fro, cos)
