"""The fused BF16 backward on networks much smaller than its 128-column operand
views (widths of 16 to 128 units on 4 to 48 inputs, layers of unequal width both
ways), against the oracle's REINFORCE gradient with the reduced-precision
bounds; and one such network's captured training step beside dense blocks."""
import numpy as np
import pytest
import torch

from oracle import estimators as est
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

from gpu_helpers import to_dev_spins

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ds,hidden,batch", [
    ((4, 30), [64, 64], 300), ((44, 48), [64, 64], 130), ((16, 33), [32, 48], 129), ((12, 48), [128, 16], 257),
    ((20, 5), [16, 128], 100), ((16, 17), [16, 32], 128), ((30, 7), [112, 64], 65)])
def test_fused_backward_small_tiles(Ds, hidden, batch):
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
    assert "bwd_fused" in model.ctx.profile_read()
    for k, D in enumerate(Ds):
        p = model.params[model.offsets[k]:model.offsets[k + 1]].cpu().numpy().astype(np.float64)
        w = est.reinforce_weights(torch.as_tensor(lz[k]), torch.as_tensor(lq[k].astype(np.float64)), model.betas[k])
        ref = est.surrogate_grad(p, D, hidden, torch.as_tensor(s[k]), w)
        g = grad[model.offsets[k]:model.offsets[k + 1]].cpu().double()
        assert torch.isfinite(g).all()
        fro = float((g - ref).norm() / ref.norm())
        cos = float(torch.nn.functional.cosine_similarity(g, ref, dim=0))
        assert fro <= 1e-1 and cos >= 0.99, (k, fro, cos)


def test_captured_step_with_small_fused_network():
    n, rest, B = 42, 12, 2246
    graphs = [wl.sk(n, 3 + k) for k in range(5)]
    Ws = [np.arange(n - rest, dtype=np.int32)] * 5
    model = TNVAN(graphs, Ws, [64, 64], [0.3 + 0.1 * k for k in range(5)], seed=1)
    step = model.capture_train_step(B, 3, tv.BF16, 0.01)
    for _ in range(4):
        step.replay()
    torch.cuda.synchronize()
    assert torch.isfinite(model.params).all() and torch.isfinite(step.stats[:, 0]).all()
