"""The FP32 backward of small networks in one kernel (at most 1,536 parameters, or at
most 450 per 64 x 64 block of weights): against
the oracle, against the general form (which a larger network beside them makes the
call take), and which of them a call launches."""
import numpy as np
import pytest
import torch

from oracle import estimators as est
from paper_2504_12037_gb300 import tnvan as tv
from paper_2504_12037_gb300 import workloads as wl
from paper_2504_12037_gb300.model import TNVAN

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]


def _model(Ds, hidden, scale=1.5):
    return TNVAN([wl.sk(D + 4, 5 + k) for k, D in enumerate(Ds)], [np.arange(D, dtype=np.int32) for D in Ds], hidden,
                 [0.7 + 0.5 * k for k in range(len(Ds))], seed=11, init_scale=scale)


def _inputs(Ds, batch, seed):
    rng = np.random.default_rng(seed)
    s = [rng.choice([-1, 1], size=(batch, D)).astype(np.int8) for D in Ds]
    return s, rng.normal(-50.0, 3.0, size=(len(Ds), batch)), rng.normal(-9.0, 1.0, size=(len(Ds), batch))


def _backward(model, s, lz, lq):
    b = lz.shape[1]
    args = (torch.as_tensor(np.concatenate([x.reshape(-1) for x in s])).cuda(), torch.as_tensor(lz.reshape(-1)).cuda(),
            torch.as_tensor(lq.astype(np.float32).reshape(-1)).cuda())
    grad = torch.full_like(model.params, float("nan"))

    def call():
        model.ctx.backward(model.betas, b, *args, tv.FP32, grad)

    call()
    torch.cuda.synchronize()
    return call, grad.cpu().double()


def _one_kernel(fn, path):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        fn()
    graph.debug_dump(str(path))
    one, two = "18bwd32_small_kernel" in path.read_text(), "18bwd32_wgrad_kernel" in path.read_text()
    assert one != two
    return one


# the smallest network, both sides of the line (1,482 and 1,560 parameters), 502 units, wide
# thin layers up to 880 units; batches of one sample, of one chunk and a sample, of chunks of 64 and a ragged one
@pytest.mark.parametrize("D,hidden,batch,one", [
    (1, [], 1, True), (38, [], 33, True), (39, [], 33, False), (1, [501], 70, True), (3, [256], 500, True),
    (400, [4], 97, True), (100, [9], 64, False), (876, [4], 40, True), (14, [17, 9], 4865, True),
    (5, [3, 2], 9999, True), (300, [1], 31, True), (2, [4, 33], 64, True)])
def test_matches_oracle(D, hidden, batch, one, tmp_path):
    Ds = [D, D]
    model = _model(Ds, hidden)
    s, lz, lq = _inputs(Ds, batch, D + batch)
    if batch == 1:
        lz[:] = lq + 3.0  # its own baseline: a zero gradient
    call, grad = _backward(model, s, lz, lq)
    assert _one_kernel(call, tmp_path / "g.dot") is one
    for k in range(2):
        p = model.params[model.offsets[k]:model.offsets[k + 1]].cpu().numpy().astype(np.float64)
        lq32 = torch.as_tensor(lq[k].astype(np.float32).astype(np.float64))
        w = est.reinforce_weights(torch.as_tensor(lz[k]), lq32, model.betas[k])
        ref = est.surrogate_grad(p, D, hidden, torch.as_tensor(s[k].astype(np.float64)), w)
        g = grad[model.offsets[k]:model.offsets[k + 1]]
        assert torch.isfinite(g).all()
        # FP32 sums of terms of the gradient's own size
        assert float((g - ref).abs().max()) <= 2e-5 * float(ref.abs().max()) + 1e-12


@pytest.mark.parametrize("D,hidden,batch", [(9, [], 20_001), (9, [16], 5_000), (6, [17, 9], 65_537)])
def test_matches_general_form(D, hidden, batch, tmp_path):
    small, mixed = _model([D, D + 3], hidden), _model([D, D + 3, 130], hidden)
    n = small.params.numel()
    assert torch.equal(small.params, mixed.params[:n])
    s, lz, lq = _inputs([D, D + 3, 130], batch, 3)
    call, a = _backward(small, s[:2], lz[:2], lq[:2])
    other, b = _backward(mixed, s, lz, lq)
    assert _one_kernel(call, tmp_path / "a.dot") and not _one_kernel(other, tmp_path / "b.dot")
    # two orders of FP32 sums of `batch` terms
    assert float((a - b[:n]).abs().max()) <= 2e-5 * float(a.abs().max())
