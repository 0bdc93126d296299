"""FP32 sampler with one and with four threads a sample: small networks over many
samples take one, and a sample's bits do not depend on it."""
import numpy as np
import pytest
import torch

from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]


def _threads(fn, path):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        fn()
    graph.debug_dump(str(path))
    one, four = "13sample_kernelILi1E" in path.read_text(), "13sample_kernelILi4E" in path.read_text()
    assert one != four
    return 1 if one else 4


@pytest.mark.parametrize("D,hidden,large", [(1, [], 65536), (6, [16], 70001), (14, [], 65536), (30, [17, 9], 80003),
                                            (30, [40], 65537), (64, [32, 48], 70000), (130, [17], 100_001)])
def test_same_bits(D, hidden, large, tmp_path):
    small, insts = 1003, 2
    graphs = [wl.sk(D + 3, 1), wl.sk(D + 3, 2)]
    model = TNVAN(graphs, [np.arange(D, dtype=np.int32)] * insts, hidden, [0.5, 1.0], seed=4, init_scale=2.0)

    def run(b):
        out = model.buffers(b)
        lq = torch.empty(insts * b, device="cuda")

        def call():
            model.ctx.sample_and_contract(model.betas, b, 21, 3, tv.FP32, *out)
            model.ctx.log_prob(b, out[0], lq, tv.FP32)

        call()
        torch.cuda.synchronize()
        spins = [model.spins_of(out[0], k, b)[:small].clone() for k in range(insts)]
        rows = [out[1][k * b:k * b + small].clone() for k in range(insts)]
        assert torch.equal(lq, out[1])  # teacher forcing on its own samples
        return _threads(call, tmp_path / f"{b}.dot"), spins, rows

    model.ctx.set_tuning((16, 0, 0, 0, 0, 0))  # 16 samples a CTA: four threads each
    t0, s0, q0 = run(small)
    model.ctx.set_tuning((0, 0, 0, 0, 0, 0))
    t1, s1, q1 = run(large)
    assert (t0, t1) == (4, 1)
    for k in range(insts):
        assert torch.equal(s0[k], s1[k]) and torch.equal(q0[k], q1[k])
