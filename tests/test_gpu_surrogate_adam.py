"""One optimiser step at a time against Adam in 64 bits: all five layers' weights and biases
with their moments, and the BF16 copies that inference and the gradients read.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_08040_gb300 import build   # noqa: E402

pytestmark = pytest.mark.gpu

ULP = 2.0 ** -24
LR, B1, B2, EPS = 3e-3, 0.9, 0.999, 1e-8


@pytest.fixture(scope="module")
def sur():
    build.build()
    from paper_2106_08040_gb300 import surrogate
    return surrogate


@pytest.mark.parametrize("steps", [1, 3])
def test_steps_follow_the_formula(sur, steps):
    """Moments within four roundings of their terms.  Weights within two roundings and 1e-4 of the update:
    1 - beta2^step, a difference of FP32 numbers near 1, is right to 2^-24 / 0.001 = 6e-5, half of
    that under the root, and the chain of quotients adds some ten roundings."""
    s = sur.Surrogate(seed=3)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)

    def fill(tensors, scale, positive=False):
        for t in tensors:
            t.copy_(torch.randn(t.shape, generator=g, device="cuda") * scale)
            if positive:
                t.abs_()

    fill(s.Wm + s.bm, 0.05)
    fill(s.mW + s.mb, 1e-3)
    fill(s.vW + s.vb, 1e-5, positive=True)
    f32 = lambda x: float(np.float32(x))            # noqa: E731  (as the call passes them)
    lr, b1, b2, eps = f32(LR), f32(B1), f32(B2), f32(EPS)
    params = list(zip(s.Wm + s.bm, s.mW + s.mb, s.vW + s.vb, s.gW + s.gb))
    for k in range(1, steps + 1):
        fill(s.gW + s.gb, 1e-2)
        before = [[t.double() for t in group] for group in params]
        s.adam(LR, B1, B2, EPS)
        torch.cuda.synchronize()
        for (p, m, v, _), (p0, m0, v0, g0) in zip(params, before):
            mr, vr = b1 * m0 + (1 - b1) * g0, b2 * v0 + (1 - b2) * g0 * g0
            assert bool(((m.double() - mr).abs() <= 4 * ULP * (m0.abs() + g0.abs())).all())
            assert bool(((v.double() - vr).abs() <= 4 * ULP * (v0 + g0 * g0)).all())
            upd = lr * (m.double() / (1 - b1 ** k)) / ((v.double() / (1 - b2 ** k)).sqrt() + eps)
            assert bool(((p.double() - (p0 - upd)).abs() <= 2 * ULP * p0.abs() + 1e-4 * upd.abs() + 1e-12).all())
            assert bool((p.double() - p0).abs().max() > 0)
        for l in range(sur.LAYERS):
            assert torch.equal(s.W[l], s.Wm[l].to(torch.bfloat16)), l
            if l > 0:
                assert torch.equal(s.WT[l], s.W[l].t()), l
    assert s.step == steps


def test_refresh_writes_the_copies_alone(sur):
    s = sur.Surrogate(seed=5)
    kept = [t.clone() for t in s.Wm + s.bm + s.mW + s.vW + s.mb + s.vb]
    for t in s.W + s.WT[1:]:
        t.fill_(float("nan"))
    s.refresh()
    for l in range(sur.LAYERS):
        assert torch.equal(s.W[l], s.Wm[l].to(torch.bfloat16)), l
        if l > 0:
            assert torch.equal(s.WT[l], s.W[l].t()), l
    assert all(torch.equal(a, b) for a, b in zip(s.Wm + s.bm + s.mW + s.vW + s.mb + s.vb, kept))
