"""Surrogate calls on workspaces of the documented sizes and on outputs of any alignment."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_08040_gb300 import build   # noqa: E402
from test_gpu_surrogate import random_net   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sur():
    build.build()
    from paper_2106_08040_gb300 import surrogate
    return surrogate


def queries(n, seed):
    return torch.from_numpy(np.random.default_rng(seed).normal(size=(n, 7)).astype(np.float32)).cuda()


@pytest.mark.parametrize("q,offset", [(1, 0), (1, 1), (3, 7), (129, 4), (700, 0), (700, 63)])
def test_ensemble_in_the_documented_workspace(sur, q, offset):
    """The mean of both networks' answers: three FP32 roundings, 2^-22 of the larger answer; nothing
    written beside the output, the spread and the workspace.  Spread: two sums of 800 squares in
    FP32, in any order (at most 160 roundings, 1e-5), here within 1e-4."""
    from paper_2106_08040_gb300 import _lib
    a, b = random_net(sur, 41), random_net(sur, 42)
    x = queries(q, 43)
    need = sum((s + 255) // 256 * 256 for s in (128 * q, 1024 * q, 1024 * q, 8 * q))
    ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    flat = torch.zeros(offset + q * 800 + 64, device="cuda")
    mean, spread = flat[offset:offset + q * 800].view(q, 800), torch.zeros(q + 1, device="cuda")
    _lib.check(_lib.lib().fp_surrogate_infer_ensemble(
        C.byref(a.net), C.byref(b.net), C.c_void_p(x.data_ptr()), q, C.c_void_p(mean.data_ptr()),
        C.c_void_p(spread.data_ptr()), C.c_void_p(ws.data_ptr()), C.c_ulonglong(need),
        C.c_void_p(a._err.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream)), "ensemble")
    y0, y1 = a.infer(x), b.infer(x)
    assert a.error_flag() == 0
    assert bool(((mean - 0.5 * (y0 + y1)).abs() <= 2.0 ** -22 * torch.maximum(y0.abs(), y1.abs())).all())
    ref = (y0 - y1).double().norm(dim=1) / (2 * mean.double().norm(dim=1))
    assert float(((spread[:q] - ref).abs() / ref).max()) <= 1e-4
    assert float(flat[:offset].abs().sum()) == 0 and float(flat[offset + q * 800:].abs().sum()) == 0
    assert float(spread[q]) == 0 and int(ws[need:].sum()) == 0


@pytest.mark.parametrize("q", [8, 264, 4096])
def test_gradients_in_the_documented_workspace(sur, q):
    """Gradients in a workspace of garbage against those in a fresh one: sums over the batch in one
    order, so the same bits; the loss is added up by atomics."""
    from paper_2106_08040_gb300 import _lib
    s = random_net(sur, 51)
    x = queries(q, 52)
    y = torch.from_numpy(np.random.default_rng(53).normal(size=(q, 800)).astype(np.float32)).cuda()
    need = sum((b + 255) // 256 * 256 for b in [128 * q] * 2 + [2048 * q, 1024 * q, 1024 * q] * 4 + [1600 * q] * 2 +
               [1024 * q] * 4)
    ws = torch.full((need + 256,), 0xC1, dtype=torch.uint8, device="cuda")
    s.grad(x, y)
    ref = [g.clone() for g in s.gW + s.gb]
    loss = float(s._loss.item())
    for g in s.gW + s.gb:
        g.fill_(float("nan"))
    _lib.check(_lib.lib().fp_surrogate_grad(
        C.byref(s.train_state), C.c_void_p(x.data_ptr()), C.c_void_p(y.data_ptr()), q, C.c_void_p(s._loss.data_ptr()),
        s._gW, s._gb, C.c_void_p(ws.data_ptr()), C.c_ulonglong(need), C.c_void_p(s._err.data_ptr()),
        C.c_void_p(torch.cuda.current_stream().cuda_stream)), "grad")
    assert s.error_flag() == 0
    assert all(torch.equal(a, b) for a, b in zip(s.gW + s.gb, ref))
    assert abs(float(s._loss.item()) - loss) <= 1e-5 * loss
    assert bool((ws[need:] == 0xC1).all())


def test_two_streams_at_one_batch_size(sur):
    """Inference, ensemble and gradients on two streams side by side repeat what they give alone."""
    from paper_2106_08040_gb300 import surrogate_train
    nets = [random_net(sur, 61), random_net(sur, 62)]
    ens = surrogate_train.Ensemble(nets)
    q = 3000
    xs = [queries(q, 63), queries(q, 64)]
    alone = [(nets[0].infer(x), ens.infer(x)[0]) for x in xs]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = [[], []]
    for i in range(30):
        for k, s in enumerate(streams):
            with torch.cuda.stream(s):
                outs[k].append(nets[0].infer(xs[k], stream=s) if i % 2 else ens.infer(xs[k], stream=s)[0])
    torch.cuda.synchronize()
    for k in range(2):
        for i, o in enumerate(outs[k]):
            assert torch.equal(o, alone[k][0] if i % 2 else alone[k][1]), (k, i)
    assert nets[0].error_flag() == 0


def test_memory_does_not_grow_with_the_batch_sizes(sur):
    s = random_net(sur, 65)
    x = queries(5000, 66)
    y = torch.empty((5000, 800), device="cuda")
    s.infer(x, out=y)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    for q in range(1000, 5000, 40):
        s.infer(x[:q], out=y[:q])
    assert torch.cuda.memory_allocated() == before
