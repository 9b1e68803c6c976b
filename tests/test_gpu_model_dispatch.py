"""Sizes on both sides of the model kernels' dispatch lines against the oracle or numpy, at
the bars of the other model tests: sums of up to a few thousand FP64 products, 1e-12
relative.
"""
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


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b))


def cplx(rng, shape):
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def dev(z):
    return torch.from_numpy(np.ascontiguousarray(np.stack([z.real, z.imag], -1))).cuda()


# one to eight narrow blocks per SM, a voxel less than the line and at it; ragged columns
@pytest.mark.parametrize("N,C,K1,Q", [(32, 1, 17, 2), (33, 1, 17, 2), (43, 1, 1000, 4), (44, 1, 1000, 4),
                                      (191, 2, 800, 4), (192, 2, 800, 4), (271, 1, 2000, 4), (272, 1, 2000, 4),
                                      (127, 1, 2500, 4), (128, 1, 2500, 4), (159, 1, 3000, 4), (160, 1, 3000, 4),
                                      (335, 1, 4200, 4), (336, 1, 4200, 4), (639, 1, 4800, 4), (640, 1, 4800, 4),
                                      (640, 1, 5000, 4)])
def test_m1_fit_at_the_lines(fp, N, C, K1, Q):
    from oracle import models
    rng = np.random.default_rng(N + Q)
    Phi, S = cplx(rng, (Q, N, C, K1)), cplx(rng, (N, C, K1))
    a = torch.empty((Q, C, K1, 2), dtype=torch.float64, device="cuda")
    eps = torch.empty((Q, C, K1), dtype=torch.float64, device="cuda")
    smax = torch.empty((C, K1), dtype=torch.float64, device="cuda")
    fp.fp_m1_fit(dev(Phi), Q, dev(S), N, C, K1, a, eps, smax)
    ag, eg = a.cpu().numpy(), eps.cpu().numpy()
    for q in (0, Q - 1):
        ao, eo = models.m1_fit(Phi[q], S)
        assert rel(ag[q][..., 0] + 1j * ag[q][..., 1], ao) <= 1e-12, q
        assert np.abs(eg[q] - eo).max() <= 1e-12 * np.abs(eo).max(), q
    np.testing.assert_allclose(smax.cpu().numpy(), np.abs(S).max(0), rtol=1e-15)


# either sum in either form: at most 128 harmonics (warps over rows), more (a thread each, 512 and 513 of them)
@pytest.mark.parametrize("A,C,K1,nk", [(1, 1, 128, 128), (1, 1, 129, 128), (1, 1, 129, 129), (3, 1, 512, 5),
                                       (40, 1, 513, 513), (17, 2, 128, 128), (2, 1, 5000, 4000), (70, 3, 130, 129)])
def test_nrmse_at_the_lines(fp, A, C, K1, nk):
    from oracle import models
    rng = np.random.default_rng(K1 + A)
    eps = rng.uniform(0.05, 0.4, size=(A, C, K1))
    ks = np.sort(rng.choice(K1, size=nk, replace=False)).astype(np.int32)
    for want in (True, False):
        ef = torch.full((K1,), np.nan, dtype=torch.float64, device="cuda") if want else None
        eg = torch.empty(1, dtype=torch.float64, device="cuda")
        fp.fp_nrmse(torch.from_numpy(eps).cuda(), A, C, K1, torch.from_numpy(ks).cuda(), nk, ef, eg)
        if want:
            assert rel(ef.cpu().numpy(), models.eps_freq(eps)) <= 1e-14
        ref = models.eps_global(eps, ks)
        assert abs(float(eg.item()) - ref) <= 1e-14 * ref


# row counts on both sides of the lines: one row group to sixteen in a block, one step of rows to several, a ragged end
@pytest.mark.parametrize("J", [16, 19, 23, 27, 31, 35, 47, 60, 63, 64, 95, 127])
@pytest.mark.parametrize("N", [85, 96, 128, 190, 512])
def test_m2_gram_at_the_lines(fp, J, N):
    A, C, K1, nk = 1, 2, 21, 16
    rng = np.random.default_rng(1000 * J + N)
    Phi, a, S = cplx(rng, (A, J, N, C, K1)), cplx(rng, (A, J, C, K1)), cplx(rng, (A, N, C, K1))
    ks = np.sort(rng.choice(K1, size=nk, replace=False)).astype(np.int32)
    smax = np.abs(S).max(1)
    G = torch.full((J + 1, J + 1, 2), np.nan, dtype=torch.float64, device="cuda")
    fp.fp_m2_gram(dev(Phi), dev(a), dev(S), torch.from_numpy(smax).cuda(), A, J, N, C, K1,
                  torch.from_numpy(ks).cuda(), nk, G)
    Gg = G.cpu().numpy()
    Gg = Gg[..., 0] + 1j * Gg[..., 1]
    M = np.concatenate([a[:, :, None] * Phi, S[:, None]], axis=1) / smax[:, None, None]
    M = M[..., ks].transpose(0, 2, 3, 4, 1).reshape(-1, J + 1)
    Go = M.conj().T @ M
    iu = np.triu_indices(J + 1)
    assert np.abs(Gg[iu] - Go[iu]).max() <= 1e-12 * np.abs(Go).max()


# 8 to 128 samples a block, ragged last blocks, fewer instances than groups of a block, a second round of them
@pytest.mark.parametrize("n,S", [(1, 4), (7, 4), (33, 4), (3000, 5), (1, 64), (40, 20), (700, 33), (130, 65),
                                 (257, 50), (3, 65), (1100, 45), (17, 816)])
def test_equilibrium_at_the_lines(fp, n, S):
    from oracle import models, physics, solve
    d = workloads.DriveSpec(amp=(0.012, 0.009, 0.0), freq=(25e3, 30e3, 0.0), phase=(np.pi / 2, 0.3, 0.0),
                            period=S / 2.5e6, samples_per_period=S, warmup_periods=1, output_periods=2)
    inst = workloads.random_instances(n, 6, seed=S)
    inst["d"] = np.random.default_rng(n).uniform(4e-9, 25e-9, n)
    inst["d"][n // 2] = 0.0                                   # no moment
    ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(), 8)
    m = torch.full((n, 2 * S, 3), np.nan, dtype=torch.float64, device="cuda")
    dm = torch.full_like(m, np.nan)
    fp.fp_equilibrium(ctx, fp.instances_to_device(inst, "cuda"), n, m, dm)
    mm, dd = m.cpu().numpy(), dm.cpu().numpy()
    assert np.isfinite(mm).all() and np.isfinite(dd).all()
    assert (mm[n // 2] == 0).all() and (dd[n // 2] == 0).all()
    drv = physics.Drive(amp=d.amp, freq=d.freq, phase=d.phase, period=d.period)
    t = solve.sample_times(drv, solve.Schedule(S, 1, 2))
    for i in sorted(({0, 1, n // 3, n - 2, n - 1} & set(range(n))) - {n // 2}):
        mo, do = models.equilibrium_trace(physics.Material(), drv, float(inst["d"][i]), inst["h_off"][i], t)
        assert rel(mm[i], mo) <= 1e-13, i
        assert rel(dd[i], do) <= 1e-12, i
    ctx.close()


# short periods of one and several channels, either side of the line between the transform and the direct sum
@pytest.mark.parametrize("S,k_max,C", [(16, 15, 1), (16, 15, 4), (24, 23, 2), (36, 35, 1), (36, 18, 4), (37, 36, 2),
                                       (37, 36, 4), (48, 24, 4), (60, 15, 1), (60, 15, 4), (64, 16, 4), (80, 20, 4)])
def test_signal_at_the_lines(fp, S, k_max, C):
    rng = np.random.default_rng(S + C)
    d = workloads.DriveSpec(amp=(0.01, 0.0, 0.0), freq=(25e3,) * 3, phase=(0.0,) * 3, period=S / 2.5e6,
                            samples_per_period=S, warmup_periods=0, output_periods=2)
    ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(), 4)
    n = 5
    dm = rng.normal(size=(n, 2 * S, 3))
    ch = rng.normal(size=(C, 3))
    out = torch.full((n, C, k_max + 1, 2), np.nan, dtype=torch.float64, device="cuda")
    fp.fp_signal(ctx, torch.from_numpy(dm).cuda(), n, k_max, ch, out)
    got = out.cpu().numpy()
    for i in range(n):
        ref = np.fft.fft(dm[i, S:] @ ch.T, axis=0).T[:, :k_max + 1] / S
        assert np.abs(got[i, ..., 0] + 1j * got[i, ..., 1] - ref).max() <= 1e-12 * np.abs(ref).max(), i
    ctx.close()
