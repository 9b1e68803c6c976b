"""Surrogate GEMM variants at the edges of their size and alignment rules.

A tile's width changes which SM forms an output, not the order of its K sum, so a
query's answer has to be the same bits in every batch: batches below and above each
threshold are compared with the leading rows of one large batch, whose answers the
oracle tests check.  Gradients are compared with the FP64 network at the bounds of the
other surrogate tests (3e-2 per tensor: BF16 activations).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_08040_gb300 import build   # noqa: E402
from test_gpu_surrogate import oracle_params, random_net, rel   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sur():
    build.build()
    from paper_2106_08040_gb300 import surrogate
    return surrogate


def thresholds():
    """Batch sizes over the range in which the tile widths change: fractions and multiples of one row block per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = [sms // 25, sms // 10, sms // 8, sms // 5, sms // 4, sms // 3, sms // 2, sms]
    return [1, 127, 257] + [128 * b + d for b in blocks for d in (0, 1)]


def queries(n, seed):
    return torch.from_numpy(np.random.default_rng(seed).normal(size=(n, 7)).astype(np.float32)).cuda()


def test_infer_is_independent_of_the_batch(sur):
    s = random_net(sur, 21)
    qs = thresholds()
    x = queries(2 * max(qs) + 77, 5)
    full = s.infer(x)
    for q in qs:
        assert torch.equal(s.infer(x[:q].contiguous()), full[:q]), q
    assert s.error_flag() == 0


@pytest.mark.parametrize("offset", [1, 4, 8])
def test_infer_into_any_alignment(sur, offset):
    s = random_net(sur, 22)
    x = queries(131, 6)
    flat = torch.zeros(131 * 800 + 64, device="cuda")
    out = flat[offset:offset + 131 * 800].view(131, 800)
    assert torch.equal(s.infer(x, out=out), s.infer(x))
    assert float(flat[:offset].abs().sum()) == 0.0 and float(flat[offset + 131 * 800:].abs().sum()) == 0.0


def test_non_finite_query_stays_in_its_row(sur):
    s = random_net(sur, 23)
    x = queries(140, 7)
    ref = s.infer(x)
    y = x.clone()
    y[3, 2], y[77, 0] = float("nan"), 3.0e38
    out = s.infer(y)
    keep = [i for i in range(140) if i not in (3, 77)]
    assert torch.equal(out[keep], ref[keep])
    assert bool(torch.isnan(out[3]).all())


def test_ensemble_is_independent_of_the_batch(sur):
    """Mean: the same bits.  Spread: two sums of 800 squares, each in 10 to 50 partial sums added in any
    order (at most 90 and 66 roundings of 2^-24 deep), under square roots: 160 roundings bound the ratio."""
    from paper_2106_08040_gb300 import surrogate_train
    ens = surrogate_train.Ensemble([random_net(sur, 31), random_net(sur, 32)])
    qs = thresholds()
    x = queries(2 * max(qs) + 77, 8)
    mean, spread = ens.infer(x)
    for q in qs:
        m, sp = ens.infer(x[:q].contiguous())
        assert torch.equal(m, mean[:q]), q
        assert float(((sp - spread[:q]).abs() / spread[:q]).max()) <= 160 * 2.0 ** -24, q


@pytest.mark.parametrize("q", [8, 4744, 9608])
def test_grad_matches_oracle_over_the_tile_rules(sur, q):
    from oracle import mlp
    s = random_net(sur, 24)
    rng = np.random.default_rng(9)
    x = rng.normal(size=(q, 7)).astype(np.float32)
    y = rng.normal(size=(q, 800)).astype(np.float32)
    loss = float(s.grad(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()).item())
    assert s.error_flag() == 0
    l_or, gW, gb = mlp.loss_and_grad(oracle_params(s), x.astype(np.float64), y.astype(np.float64))
    assert abs(loss - l_or) / l_or < 1e-2
    for l in range(sur.LAYERS):
        assert rel(s.gW[l].cpu().numpy(), gW[l]) < 3e-2, l
        assert rel(s.gb[l].cpu().numpy(), gb[l]) < 3e-2, l


def test_launches_can_be_captured(sur):
    """The overlapped launches of an inference, recorded into a CUDA graph, answer new inputs on replay."""
    s = random_net(sur, 25)
    x = queries(300, 10)
    y = torch.empty((300, 800), device="cuda")
    s.infer(x, out=y)                                  # workspace and module load happen outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.infer(x, out=y)
    x2 = queries(300, 11)
    ref = s.infer(x2)
    x.copy_(x2)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, ref) and s.error_flag() == 0
