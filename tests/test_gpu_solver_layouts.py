"""Five-stage solves with the factors in shared memory (batches of at most one
instance per SM) against the two-CTA layout with factors in global memory.

Both layouts do the same operations on an instance, so a batch of one instance more,
which takes the other layout, has to repeat the answers.  Asserted is what each of the two is
held to against the oracle: traces within 1e-9 of the solution, hence 2e-9 of each
other, and their derivatives within the 1e-6 that the l = 1 rows of the operator make of it.
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


@pytest.mark.parametrize("L_launch,L_lo,L_hi", [(2, 2, 2), (9, 6, 9), (16, 10, 16)])
def test_shared_memory_factors_repeat_the_global_ones(fp, L_launch, L_lo, L_hi):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    d = workloads.DriveSpec(amp=(0.004, 0.002, 0.0), freq=(50e3,) * 3, phase=(0.0, 0.7, 0.0), period=2e-5,
                            samples_per_period=12, warmup_periods=0, output_periods=1)
    ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(rtol=1e-10, stages=5), L_launch)
    inst = workloads.random_instances(sms + 1, max(L_launch, 6), seed=5, max_offset=0.002, K_range=(1e2, 5e2))
    inst["L"] = np.random.default_rng(6).integers(L_lo, L_hi + 1, sms + 1)
    inst["L"][3] = L_launch + 1                      # refused in either layout
    out = {}
    for n in (1, sms, sms + 1):
        out[n] = [a.cpu().numpy() for a in fp.solve(ctx, inst[:n])]
    ctx.close()
    m, dm, st, stats = out[sms + 1]
    for n in (1, sms):
        assert (out[n][2] == st[:n]).all() and (out[n][3][:, 0] == stats[:n, 0]).all()
        for a, b, bar in ((out[n][0], m[:n], 2e-9), (out[n][1], dm[:n], 2e-6)):
            assert np.linalg.norm(a - b) <= bar * np.linalg.norm(b)
    assert st[3] == 5 and (m[3] == 0).all()          # FP_STATUS_BAD_INPUT
