"""Edges of the model kernels' size rules (fp_signal, fp_equilibrium, fp_m1_fit,
fp_nrmse, fp_m2_gram) against the FP64 oracle or numpy, at the bars of the model tests:
sums of up to a few thousand FP64 products, 1e-12 relative (1e-13 for <m> of M0).
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


def schedule(S, W=0):
    return workloads.DriveSpec(amp=(0.012, 0.009, 0.0), freq=(25e3, 30e3, 0.0), phase=(np.pi / 2, 0.3, 0.0),
                               period=S / 2.5e6, samples_per_period=S, warmup_periods=W, output_periods=2)


# primes (one radix), powers, three radices, few harmonics and long periods (direct sum)
@pytest.mark.parametrize("S,k_max,C,shift", [
    (2, 1, 1, 0), (3, 2, 2, 0), (4, 3, 1, 0), (17, 16, 2, 0), (64, 63, 3, 0), (101, 50, 2, 0), (101, 100, 1, 0),
    (204, 102, 4, 0), (1632, 816, 2, 0), (1632, 1631, 1, 0), (1632, 0, 1, 0), (1632, 5, 2, 0), (1632, 816, 1, 1),
    (2520, 1260, 1, 0), (4098, 4097, 1, 0), (6000, 40, 2, 0), (3999, 3998, 1, 0)])
def test_signal_sizes(fp, S, k_max, C, shift):
    """shift = 1: the result starts 8 bytes off a 16-byte boundary.  Reference:
    numpy's FFT (8e-18 from a long-double sum at S = 3999, k = 3998, where the
    oracle's angles 2 pi j k / S, unreduced, are 2.9e-14 off)."""
    rng = np.random.default_rng(S + k_max)
    ctx = fp.Context(fp.Material(), fp.Drive(**schedule(S).__dict__), fp.Tol(), 4)
    n = 3
    dm = rng.normal(size=(n, 2 * S, 3))
    ch = rng.normal(size=(C, 3))
    buf = torch.full((n * C * (k_max + 1) * 2 + 1,), np.nan, dtype=torch.float64, device="cuda")
    out = buf[shift:shift + n * C * (k_max + 1) * 2].view(n, C, k_max + 1, 2)
    fp.fp_signal(ctx, torch.from_numpy(dm).cuda(), n, k_max, ch, out)
    got = out.cpu().numpy()
    for i in range(n):
        ref = np.fft.fft(dm[i, S:] @ ch.T, axis=0).T[:, :k_max + 1] / S
        assert np.abs(got[i, ..., 0] + 1j * got[i, ..., 1] - ref).max() <= 1e-12 * np.abs(ref).max(), i
    ctx.close()


@pytest.mark.parametrize("n,S", [(1, 2), (1, 129), (17, 128), (700, 300)])
def test_equilibrium_sizes(fp, n, S):
    from oracle import models, physics, solve
    d = schedule(S, W=1)
    inst = workloads.random_instances(n, 6, seed=S)
    inst["d"] = np.random.default_rng(n).uniform(4e-9, 25e-9, n)      # Langevin arguments on both sides of the series
    ctx = fp.Context(fp.Material(), fp.Drive(**d.__dict__), fp.Tol(), 8)
    m = torch.full((n, 2 * S, 3), np.nan, dtype=torch.float64, device="cuda")
    dm = torch.full_like(m, np.nan)
    fp.fp_equilibrium(ctx, fp.instances_to_device(inst, "cuda"), n, m, dm)
    mm, dd = m.cpu().numpy(), dm.cpu().numpy()
    assert np.isfinite(mm).all() and np.isfinite(dd).all()
    drv = physics.Drive(amp=d.amp, freq=d.freq, phase=d.phase, period=d.period)
    t = solve.sample_times(drv, solve.Schedule(S, 1, 2))
    for i in sorted({0, n // 2, n - 1}):
        mo, do = models.equilibrium_trace(physics.Material(), drv, float(inst["d"][i]), inst["h_off"][i], t)
        assert rel(mm[i], mo) <= 1e-13, i
        assert rel(dd[i], do) <= 1e-12, i
    ctx.close()


# narrow blocks (ragged columns, fewer voxels than groups) and wide ones
@pytest.mark.parametrize("N,C,K1,Q", [(31, 1, 17, 2), (1, 1, 1, 1), (33, 1, 1000, 20), (5, 2, 65, 120)])
def test_m1_fit_block_shapes(fp, N, C, K1, Q):
    from oracle import models
    rng = np.random.default_rng(N * Q)
    Phi, S = cplx(rng, (Q, N, C, K1)), cplx(rng, (N, C, K1))
    a = torch.empty((Q, C, K1, 2), dtype=torch.float64, device="cuda")
    eps = torch.empty((Q, C, K1), dtype=torch.float64, device="cuda")
    smax = torch.empty((C, K1), dtype=torch.float64, device="cuda")
    fp.fp_m1_fit(dev(Phi), Q, dev(S), N, C, K1, a, eps, smax)
    ag, eg = a.cpu().numpy(), eps.cpu().numpy()
    for q in sorted({0, Q // 2, Q - 1}):
        ao, eo = models.m1_fit(Phi[q], S)
        assert rel(ag[q][..., 0] + 1j * ag[q][..., 1], ao) <= 1e-12, q
        assert np.abs(eg[q] - eo).max() <= 1e-12 * max(np.abs(eo).max(), 1e-2), q
    np.testing.assert_allclose(smax.cpu().numpy(), np.abs(S).max(0), rtol=1e-15)


@pytest.mark.parametrize("A,C,K1,nk", [(1, 1, 1, 1), (12, 3, 128, 7), (33, 1, 129, 129), (5, 2, 300, 131)])
def test_nrmse_sizes(fp, A, C, K1, nk):
    from oracle import models
    rng = np.random.default_rng(K1)
    eps = rng.uniform(0.05, 0.4, size=(A, C, K1))
    ks = np.sort(rng.choice(K1, size=nk, replace=False)).astype(np.int32)
    for want in (True, False):
        ef = torch.empty(K1, dtype=torch.float64, device="cuda") if want else None
        eg = torch.empty(1, dtype=torch.float64, device="cuda")
        fp.fp_nrmse(torch.from_numpy(eps).cuda(), A, C, K1, torch.from_numpy(ks).cuda(), nk, ef, eg)
        if want:
            assert rel(ef.cpu().numpy(), models.eps_freq(eps)) <= 1e-14
        ref = models.eps_global(eps, ks)
        assert abs(float(eg.item()) - ref) <= 1e-14 * ref


# tiled kernel (few columns, many columns, few rows), micro tiles with and without several row groups
@pytest.mark.parametrize("A,J,N,C,K1,nk", [(2, 15, 60, 2, 12, 11), (2, 16, 60, 2, 12, 11), (1, 17, 97, 1, 30, 23),
                                           (3, 40, 40, 2, 12, 11), (2, 96, 61, 2, 12, 9), (2, 127, 61, 2, 12, 9),
                                           (2, 128, 61, 2, 12, 9), (1, 30, 19, 1, 40, 23)])
def test_m2_gram_shapes(fp, A, J, N, C, K1, nk):
    rng = np.random.default_rng(A * 1000 + J)
    Phi, a, S = cplx(rng, (A, J, N, C, K1)), cplx(rng, (A, J, C, K1)), cplx(rng, (A, N, C, K1))
    ks = np.sort(rng.choice(K1, size=nk, replace=False)).astype(np.int32)
    smax = np.abs(S).max(1)
    smax[0, 0, ks[0]] = 0.0                                   # this row is dropped
    G = torch.full((J + 1, J + 1, 2), np.nan, dtype=torch.float64, device="cuda")
    fp.fp_m2_gram(dev(Phi), dev(a), dev(S), torch.from_numpy(smax).cuda(), A, J, N, C, K1,
                  torch.from_numpy(ks).cuda(), nk, G)
    Gg = G.cpu().numpy()
    Gg = Gg[..., 0] + 1j * Gg[..., 1]
    with np.errstate(divide="ignore"):
        sig = np.where(smax > 0, 1.0 / smax, 0.0)
    M = np.concatenate([a[:, :, None] * Phi, S[:, None]], axis=1) * sig[:, None, None]
    M = M[..., ks].transpose(0, 2, 3, 4, 1).reshape(-1, J + 1)
    Go = M.conj().T @ M
    iu = np.triu_indices(J + 1)
    assert np.abs(Gg[iu] - Go[iu]).max() <= 1e-12 * np.abs(Go).max()
