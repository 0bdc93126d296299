"""Autotuning does not lose the launch shapes the library picks by batch size."""
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

pytestmark = pytest.mark.gpu


def _time(fn):
    for _ in range(3):
        fn()
    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_autotuned_fp32_sampler_keeps_its_rule():
    """5 x 4,099 samples: 148 us by the rule (one wave of CTAs), 211 with 16 samples a CTA, the fastest of the
    fixed counts."""
    insts, B = 5, 4099
    gs = [wl.lattice(16, 16, "gauss", 5 + k) for k in range(insts)]
    model = TNVAN(gs, [wl.width_columns(16, 16, [3, 7, 11, 15])] * insts, [128, 128], [0.9] * insts, seed=1)
    out = model.buffers(B)

    def call():
        model.ctx.sample_and_contract(model.betas, B, 3, 1, tv.FP32, *out)

    before = _time(call)
    choice = model.ctx.autotune(model.betas, B, tv.FP32)
    assert choice[0] in (16, 32, 64) and choice[1] in (32, 64, 128)
    assert _time(call) <= 1.15 * before
