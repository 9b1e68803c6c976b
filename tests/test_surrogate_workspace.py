"""Workspace sizes of the surrogate calls (host only): what a query takes, so that a caller's
buffer of this size stays large enough.  Each array is rounded up to 256 bytes.
"""
import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2106_08040_gb300 import build
    build.build()
    from paper_2106_08040_gb300 import _lib
    return _lib.lib()


def total(*sizes):
    return sum((s + 255) // 256 * 256 for s in sizes)


@pytest.mark.parametrize("q", [1, 7, 257, 4096, 1024000])
def test_inference_and_ensemble(lib, q):
    x0, h = 128 * q, 1024 * q                        # bf16 inputs (64 wide) and activations (512 wide)
    assert lib.fp_surrogate_workspace_bytes(q, 0) <= total(x0, h, h)
    assert lib.fp_surrogate_workspace_bytes(q, 2) <= total(x0, h, h, 8 * q)


@pytest.mark.parametrize("q", [8, 64, 4096, 65536])
def test_training(lib, q):
    """bf16 inputs and their transpose; per hidden layer FP32 pre-activations, activations and their
    transpose; output cotangents and their transpose; two pairs of hidden cotangents."""
    layer = [2048 * q, 1024 * q, 1024 * q]
    assert lib.fp_surrogate_workspace_bytes(q, 1) <= total(128 * q, 128 * q, *layer * 4, 1600 * q, 1600 * q,
                                                           *[1024 * q] * 4)
