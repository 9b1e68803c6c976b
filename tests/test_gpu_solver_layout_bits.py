"""A five-stage instance gives the same bits in a batch of one, of one per SM (factors in
shared memory, one CTA per SM) and of one more (factors in global memory, two CTAs per
SM): traces, derivatives, status and all four statistics.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_08040_gb300 import build, workloads   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    build.build()
    from paper_2106_08040_gb300 import fp
    return fp


@pytest.mark.parametrize("L_launch,L_lo", [(2, 2), (3, 2), (9, 6), (16, 10)])
def test_layouts_agree_bit_for_bit(fp, L_launch, L_lo):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d = workloads.DriveSpec(amp=(0.008, 0.005, 0.0), freq=(50e3, 47e3, 50e3), phase=(0.0, 0.7, 0.0), period=2e-5,
                            samples_per_period=10, warmup_periods=0, output_periods=1)
    ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(rtol=1e-9, stages=5), L_launch)
    inst = workloads.random_instances(sms + 1, L_launch, seed=17, K_range=(1e2, 4e3))
    inst["L"] = np.random.default_rng(18).integers(L_lo, L_launch + 1, sms + 1)
    inst["L"][5] = 1                                  # refused in either layout
    full = fp.solve(ctx, inst)
    for n in (1, sms):
        for a, b in zip(fp.solve(ctx, inst[:n]), full):
            assert torch.equal(a, b[:n]), n
    ctx.close()
