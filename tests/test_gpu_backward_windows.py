"""The FP32 backward takes a large batch in windows of bounded memory: the same
gradient as its parts, a last ragged window included, and no workspace that grows
with the batch."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

pytestmark = pytest.mark.gpu


def _model():
    # 2 (8 + 64 + 64) rows a sample: windows of 986,880 samples
    return TNVAN([wl.sk(20, 3)], [np.arange(8, dtype=np.int32)], [64, 64], [0.7], seed=5)


def _batch(b, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = (torch.randint(0, 2, (b * 8,), device="cuda", dtype=torch.int8, generator=gen) * 2 - 1)
    lz = torch.randn(b, device="cuda", dtype=torch.float64, generator=gen) * 3
    lq = torch.randn(b, device="cuda", generator=gen)
    return s, lz, lq


def test_windows_add_up():
    model, b = _model(), 1_000_003
    s, lz, lq = _batch(b, 1)
    full, part, total = (torch.zeros_like(model.params) for _ in range(3))
    model.ctx.backward(model.betas, b, s, lz, lq, tv.FP32, full)
    model.ctx.reduce(model.betas, b, lz, lq)  # the baseline and batch size of the whole batch
    for lo, hi in ((0, 500_000), (500_000, b)):
        model.ctx.backward_stats(model.betas, hi - lo, s[8 * lo:8 * hi].clone(), lz[lo:hi].clone(), lq[lo:hi].clone(),
                                 tv.FP32, part)
        total += part
    torch.cuda.synchronize()
    # FP32 sums of 1e6 terms in slices of a few thousand
    assert float((full - total).abs().max()) <= 1e-5 * float(full.abs().max())


def test_workspace_does_not_grow_with_the_batch():
    model, rep = _model(), 16
    s, lz, lq = _batch(1 << 18, 2)
    one, many = torch.zeros_like(model.params), torch.zeros_like(model.params)
    model.ctx.backward(model.betas, 1 << 18, s, lz, lq, tv.FP32, one)
    s, lz, lq = s.repeat(rep), lz.repeat(rep), lq.repeat(rep)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    model.ctx.backward(model.betas, rep << 18, s, lz, lq, tv.FP32, many)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 1.3e9  # 4.6e9 in one piece
    assert float((one - many).abs().max()) <= 1e-5 * float(one.abs().max())
