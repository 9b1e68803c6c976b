"""Calls from several host threads at once, each thread with its own buffers, stream and
(where the call takes one) context: a kernel's dynamic shared-memory limit is state of the
process, so a launch must not depend on the size that another thread asks for in between.
Refusals would come back as errors of the launch; nothing here faults.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2106_08040_gb300 import build, workloads      # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    build.build()
    from paper_2106_08040_gb300 import fp as fpmod
    return fpmod


def run_threads(calls, repeat, sync_every):
    """Each call, a function of a stream, `repeat` times in a thread of its own; the errors raised.
    A full launch queue would hold the threads back, so each waits for its stream now and then."""
    errors = []
    start = threading.Barrier(len(calls))

    def loop(call):
        s = torch.cuda.Stream()
        start.wait()
        for i in range(repeat):
            try:
                call(s)
            except RuntimeError as e:
                errors.append(str(e))
            if i % sync_every == sync_every - 1:
                s.synchronize()
        s.synchronize()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=loop, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def test_m2_gram_of_different_column_counts(fp):
    def call(J, N=64, nk=32):
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")        # noqa: E731
        ks = torch.arange(nk, dtype=torch.int32, device="cuda")
        a = (z(1, J, N, 1, nk, 2), z(1, J, 1, nk, 2), z(1, N, 1, nk, 2), z(1, 1, nk) + 1.0, 1, J, N, 1, nk, ks, nk,
             z(J + 1, J + 1, 2))
        return lambda s: fp.fp_m2_gram(*a, stream=s)

    assert run_threads([call(J) for J in (35, 48) * 3], 20000, 1) == []


@pytest.mark.parametrize("stages,n,degrees", [(3, 1, (4, 16)), (5, 1, (4, 16)), (5, 200, (4, 16)), (3, 1, (17, 24))])
def test_solves_of_different_degrees(fp, stages, n, degrees):
    """Instances of no volume: every launch ends at once, with status FP_STATUS_BAD_INPUT."""
    d = workloads.DriveSpec(amp=(0.01, 0.0, 0.0), freq=(25e3,) * 3, phase=(0.0,) * 3, period=4e-5,
                            samples_per_period=2, warmup_periods=0, output_periods=1)
    ctxs, statuses = [], []

    def call(L):
        ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(stages=stages), L)
        inst = workloads.random_instances(n, L)
        inst["d"] = 0.0
        d_inst = fp.instances_to_device(inst)
        st = torch.zeros(n, dtype=torch.int32, device="cuda")
        ctxs.append(ctx)
        statuses.append(st)
        return lambda s: fp.fp_solve_batch(ctx, d_inst, n, None, None, st, None, stream=s)

    assert run_threads([call(L) for L in degrees * 3], 3000, 250) == []
    assert all(bool((st == 5).all()) for st in statuses)
    for c in ctxs:
        c.close()


def test_signals_of_different_periods(fp):
    """Two harmonics of periods of 32 and 20,000 samples: the direct sum, whose samples lie in shared memory."""
    ctxs = []

    def call(S):
        d = workloads.DriveSpec(amp=(0.01, 0.0, 0.0), freq=(25e3,) * 3, phase=(0.0,) * 3, period=S / 2.5e6,
                                samples_per_period=S, warmup_periods=0, output_periods=1)
        ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(), 4)
        ctxs.append(ctx)
        dm = torch.ones((1, S, 3), dtype=torch.float64, device="cuda")
        out = torch.empty((1, 1, 2, 2), dtype=torch.float64, device="cuda")
        ch = np.array([[1.0, 0.0, 0.0]])
        return lambda s: fp.fp_signal(ctx, dm, 1, 1, ch, out, stream=s)

    assert run_threads([call(S) for S in (32, 20000) * 3], 1500, 250) == []
    for c in ctxs:
        c.close()
