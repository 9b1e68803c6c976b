"""Performance cases of the framework: what its users have it do, through its public entry points.

A case is a dict of plain values with a "kind":

  solve     fp_solve_batch: <m>(t) and d<m>/dt(t) of a batch of instances of uneven degree
  sysmat    fp_solve_batch + fp_signal: phi_hat of a voxel grid (one column of a system matrix per voxel)
  sweep     fp_sweep_plan / fp_sweep_run: a parameter sweep over degrees 8..24, traces of every draw
  grad      fp.phi_hat and its backward pass: misfit and gradient of candidate parameter sets on a voxel grid
  ensemble  Ensemble.infer: surrogate answer and spread, two networks
  infer     Surrogate.infer: one network
  train     Surrogate.grad + Surrogate.adam: one optimiser step
  m0        fp_equilibrium + fp_signal: model M0 traces and phi_hat
  m1        fp_m1_fit + fp_nrmse: filter fit of a dictionary and its distance measures
  m2        fp_m2_gram: Gram matrix of the weighted dictionary

Schedules keep the x frequency of the benchmark drive (2.5 MHz / 102) and take the y frequency as
(density + 1) / density of it, so one Lissajous period holds 102 * density samples at 2.5 MHz
(density 16 is the benchmark's 1632-sample period).
"""
import math
import os

import numpy as np
import torch

from paper_2106_08040_gb300 import fp, surrogate, surrogate_train, workloads

DEV = "cuda"
CH = [[1.0, 0.0, 0.0], [0.0, 1.0, 0.0]]
DATA = os.path.join(os.path.dirname(os.path.abspath(surrogate_train.__file__)), "data", "surrogate_L16")
KB = 1.380649e-23


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # one particle ensemble looked at by hand: the single-instance workload's degree and drive, one period
        {"name": "trace_one_L10", "kind": "solve", "n": 1, "L_min": 10, "L_max": 10, "stages": 5, "rtol": 1e-9,
         "samples": 1000, "drive": "sine"},
        # a few hundred random ensembles, degree by the truncation rule, two waves of CTAs
        {"name": "traces_301_ragged", "kind": "solve", "n": 301, "L_min": 8, "L_max": 16, "stages": 3, "rtol": 1e-10,
         "samples": 64, "drive": "xy"},
        # a patch of the system matrix with the full 1632-sample period: fewer voxels than the GPU has SMs
        {"name": "sysmat_60_full_period", "kind": "sysmat", "nx": 10, "ny": 6, "L": 16, "stages": 5, "rtol": 1e-9,
         "density": 16, "warmup": 0},
        # the benchmark's 32 x 32 grid at degree 16, warm-up and output period, on a coarser Lissajous curve
        {"name": "sysmat_1024", "kind": "sysmat", "nx": 32, "ny": 32, "L": 16, "stages": 5, "rtol": 1e-9,
         "density": 2, "warmup": 1},
        # parameter sweep over stiffness and degree, one plan and one submission
        {"name": "sweep_257_L8_24", "kind": "sweep", "n": 257, "L_min": 8, "L_max": 24, "bucket": 2, "rtol": 1e-9,
         "density": 1},
        # one iteration of an adjoint-driven fit: a candidate set over a 10 x 10 voxel grid
        {"name": "fit_gradient_100", "kind": "grad", "sets": 1, "nx": 10, "ny": 10, "L": 16, "rtol": 1e-9,
         "density": 1, "k_max": 50},
        # the surrogate grid: 40 x 40 x 40 offsets x 16 easy axes, two networks
        {"name": "surrogate_ensemble_1m", "kind": "ensemble", "q": 1024000},
        # a handful of queries, where launches count
        {"name": "surrogate_infer_257", "kind": "infer", "q": 257},
        # one training step at the default batch
        {"name": "surrogate_train_4096", "kind": "train", "q": 4096},
        # equilibrium model of the whole grid at the benchmark's period, up to the Nyquist row
        {"name": "m0_phihat_1024", "kind": "m0", "nx": 32, "ny": 32, "density": 16, "warmup": 1, "k_max": 816},
        # M1 fit of 8 diameters x 12 anisotropies against one measured matrix
        {"name": "m1_fit_96", "kind": "m1", "Q": 96, "N": 1024, "C": 2, "K1": 817, "orders": 20},
        # M2 dictionary of 96 tuples over 12 angles on an 11 x 11 grid
        {"name": "m2_gram_96", "kind": "m2", "A": 12, "J": 96, "N": 121, "C": 2, "K1": 817, "orders": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "sysmat", "sweep", "grad", "ensemble", "infer", "train", "m0", "m1", "m2"])
    if kind == "solve":
        lo = rng.randint(6, 12)
        return {"kind": kind, "n": _log(rng, 1, 700), "L_min": lo, "L_max": rng.randint(max(lo, 10), 16),
                "stages": rng.choice([3, 5]), "rtol": rng.choice([1e-9, 1e-10]), "samples": _log(rng, 40, 160),
                "drive": rng.choice(["sine", "xy"])}
    if kind == "sysmat":
        # intervals x waves of resident instances stay below the 32 x 32 case
        density = rng.choice([1, 2, 5])
        side = {1: 32, 2: 24, 5: 17}[density]
        return {"kind": kind, "nx": _log(rng, 2, side), "ny": _log(rng, 2, side), "L": rng.randint(10, 16),
                "stages": rng.choice([3, 5]), "rtol": 1e-9, "density": density, "warmup": rng.choice([0, 1])}
    if kind == "sweep":
        return {"kind": kind, "n": _log(rng, 16, 300), "L_min": 8, "L_max": rng.choice([16, 20, 24]),
                "bucket": rng.choice([1, 2, 4]), "rtol": 1e-9, "density": 1}
    if kind == "grad":
        return {"kind": kind, "sets": rng.randint(1, 3), "nx": rng.randint(2, 7), "ny": rng.randint(2, 7),
                "L": rng.randint(8, 16), "rtol": 1e-9, "density": 1, "k_max": _log(rng, 8, 100)}
    if kind in ("ensemble", "infer"):
        return {"kind": kind, "q": _log(rng, 1, 700000)}
    if kind == "train":
        return {"kind": kind, "q": 8 * _log(rng, 1, 2048)}
    if kind == "m0":
        density = rng.choice([1, 2, 5, 16])
        return {"kind": kind, "nx": _log(rng, 2, 32), "ny": _log(rng, 2, 32), "density": density,
                "warmup": rng.choice([0, 1]), "k_max": _log(rng, 8, 102 * density - 1)}
    if kind == "m1":
        return {"kind": kind, "Q": _log(rng, 1, 96), "N": _log(rng, 16, 1024), "C": rng.choice([1, 2, 3]),
                "K1": _log(rng, 40, 500), "orders": rng.choice([5, 10, 20])}
    return {"kind": kind, "A": rng.randint(1, 12), "J": _log(rng, 2, 96), "N": _log(rng, 9, 121),
            "C": rng.choice([1, 2]), "K1": _log(rng, 40, 817), "orders": rng.choice([5, 10, 20])}


# ------------------------------------------------------------------ inputs --
def _lissajous(density, warmup):
    n = density
    return workloads.DriveSpec(amp=(0.012, 0.012, 0.0), freq=(2.5e6 / 102.0, 2.5e6 * (n + 1) / (102.0 * n), 0.0),
                               phase=(np.pi / 2, np.pi / 2, 0.0), period=102 * n / 2.5e6,
                               samples_per_period=102 * n, warmup_periods=warmup, output_periods=1)


def _drive(dspec):
    return fp.Drive(**dspec.__dict__)


def _rule_degrees(inst, dspec, lo, hi):
    inst["L"] = fp.truncation_degree(inst, drive=_drive(dspec), L_min=lo, L_max=hi)
    return inst


def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _grid(case, seed, L):
    """A voxel grid of the benchmark's field of view with one (angle, K, d) tuple per seed."""
    rng = np.random.default_rng(seed)
    inst = workloads.make_instances(case["nx"] * case["ny"])
    inst["h_off"] = workloads.voxel_offsets(case["nx"], case["ny"])
    inst["theta"] = np.pi / 2
    inst["phi"] = rng.uniform(0.0, np.pi)
    inst["K"] = rng.uniform(1.5e3, 2.5e3)
    inst["d"] = rng.uniform(18.5e-9, 20.5e-9)
    inst["L"] = L
    return inst


def _queries(case, seed):
    """Surrogate inputs: draws of its training distribution."""
    inst = workloads.uneven_sweep_instances(case["q"], 16, seed=seed)
    return torch.from_numpy(surrogate.features(inst).astype(np.float32)).to(DEV)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _matrix(shape, K1, g):
    """Synthetic phi_hat-like complex data [..., K1, 2]: harmonics that fall off with k."""
    x = torch.randn(tuple(shape) + (K1, 2), dtype=torch.float64, device=DEV, generator=g)
    env = 1.0 / (1.0 + torch.arange(K1, dtype=torch.float64, device=DEV) / 20.0) ** 2
    return x.mul_(env[:, None])


def _cplx(x):
    return torch.view_as_complex(x)


def _ks(case):
    return torch.from_numpy(fp.fp_freq_index_set(case["orders"], case["orders"], 16, case["K1"] - 1)).to(DEV)


def _m1_data(case, seed):
    g = _gen(seed)
    Q, N, C, K1 = case["Q"], case["N"], case["C"], case["K1"]
    phi = _matrix((Q, N, C), K1, g)
    filt = torch.randn((C, K1, 2), dtype=torch.float64, device=DEV, generator=g)
    S = torch.view_as_real(_cplx(filt) * _cplx(phi[0])).contiguous()      # a filter on the first element, 5 % noise
    S += 0.05 * S.abs().mean(dim=(0, 1, 3), keepdim=True) * torch.randn(S.shape, dtype=S.dtype, device=DEV, generator=g)
    return phi, S


def _m2_data(case, seed):
    g = _gen(seed)
    A, J, N, C, K1 = case["A"], case["J"], case["N"], case["C"], case["K1"]
    phi = _matrix((A, J, N, C), K1, g)
    a = torch.randn((A, J, C, K1, 2), dtype=torch.float64, device=DEV, generator=g)
    w = torch.rand((J,), dtype=torch.float64, device=DEV, generator=g)
    S = _empty(A, N, C, K1, 2)
    for t in range(A):                                                     # superposition of the dictionary, 5 % noise
        s = torch.zeros((N, C, K1), dtype=torch.complex128, device=DEV)
        for j in range(J):
            s += w[j] * _cplx(a[t, j]) * _cplx(phi[t, j])
        S[t] = torch.view_as_real(s)
    S += 0.05 * S.abs().mean() * torch.randn(S.shape, dtype=S.dtype, device=DEV, generator=g)
    smax = S.square().sum(-1).sqrt().amax(1).contiguous()
    return phi, a, S, smax


def _train_data(case, seed):
    """Inputs of the training distribution and targets of a signal's size around the output normalisation."""
    z = np.load(DATA + ".m0.npz")
    x = _queries(case, seed)
    g = _gen(seed)
    y = torch.randn((case["q"], surrogate.N_OUT), device=DEV, generator=g)
    y = y * torch.from_numpy(z["out_scale"]).to(DEV) + torch.from_numpy(z["out_shift"]).to(DEV)
    return x, y


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "solve":
        rng = np.random.default_rng(seed)
        S = case["samples"]
        if case["drive"] == "sine":
            d = workloads.DriveSpec(amp=(0.012, 0.0, 0.0), freq=(25e3,) * 3, phase=(0.0,) * 3, period=4e-5,
                                    samples_per_period=S, warmup_periods=0, output_periods=1)
        else:
            d = workloads.DriveSpec(amp=(0.010, 0.004, 0.0), freq=(50e3,) * 3, phase=(0.0, 0.7, 0.0), period=2e-5,
                                    samples_per_period=S, warmup_periods=0, output_periods=1)
        inst = workloads.random_instances(case["n"], 10, seed=int(rng.integers(1 << 31)), max_offset=0.004,
                                          K_range=(5e2, 3e3))
        inst = _rule_degrees(inst, d, case["L_min"], case["L_max"])
        s["ctx"] = fp.Context(fp.Material(), _drive(d), fp.Tol(rtol=case["rtol"], stages=case["stages"]), case["L_max"])
        s["inst"] = fp.instances_to_device(inst, DEV)
        s["m"], s["dm"] = _empty(case["n"], S, 3), _empty(case["n"], S, 3)
        s["st"] = _empty(case["n"], dtype=torch.int32)
    elif kind == "sysmat":
        d = _lissajous(case["density"], case["warmup"])
        inst = _grid(case, seed, case["L"])
        s["n"], s["k_max"] = len(inst), d.samples_per_period // 2
        s["ctx"] = fp.Context(fp.Material(), _drive(d), fp.Tol(rtol=case["rtol"], stages=case["stages"]), case["L"])
        s["inst"] = fp.instances_to_device(inst, DEV)
        s["dm"] = _empty(s["n"], d.samples_per_period, 3)
        s["st"] = _empty(s["n"], dtype=torch.int32)
        s["ph"] = _empty(s["n"], 2, s["k_max"] + 1, 2)
    elif kind == "sweep":
        d = _lissajous(case["density"], 0)
        pool = workloads.uneven_sweep_instances(4 * case["n"] + 64, 8, seed=seed)
        keep = fp.Material().sigma(pool["K"], pool["d"]) <= 12.0            # barriers that these degrees resolve
        inst = _rule_degrees(pool[keep][:case["n"]].copy(), d, case["L_min"], case["L_max"])
        s["n"] = len(inst)
        s["ctx"] = fp.Context(fp.Material(), _drive(d), fp.Tol(rtol=case["rtol"], stages=3), case["L_max"])
        s["inst"] = fp.instances_to_device(inst, DEV)
        s["sw"] = fp.Sweep(s["ctx"], inst, bucket_width=case["bucket"])
        s["stream"] = torch.cuda.Stream()
        s["m"], s["dm"] = (_empty(s["n"], d.samples_per_period, 3) for _ in range(2))
        s["st"] = _empty(s["n"], dtype=torch.int32)
    elif kind == "grad":
        d = _lissajous(case["density"], 0)
        rng = np.random.default_rng(seed)
        P, off = case["sets"], workloads.voxel_offsets(case["nx"], case["ny"])
        p = np.column_stack([rng.uniform(1.5e3, 2.5e3, P), rng.uniform(18.5e-9, 20.5e-9, P),
                             rng.uniform(1.0, 2.0, P), rng.uniform(0.0, np.pi, P)])
        s["ctx"] = fp.Context(fp.Material(), _drive(d), fp.Tol(rtol=case["rtol"], stages=3, max_steps=20000), case["L"])
        s["params"] = torch.from_numpy(np.repeat(p, len(off), axis=0)).to(DEV)
        s["h_off"] = torch.from_numpy(np.tile(off, (P, 1))).to(DEV)
        s["u"] = 1e4 * _matrix((P * len(off), 2), case["k_max"] + 1, _gen(seed))
    elif kind == "ensemble":
        s["net"] = surrogate_train.Ensemble.load(DATA + ".npz")
        s["x"] = _queries(case, seed)
    elif kind == "infer":
        s["net"] = surrogate.Surrogate.load(DATA + ".m0.npz")
        s["x"] = _queries(case, seed)
    elif kind == "train":
        s["net"] = surrogate.Surrogate.load(DATA + ".m0.npz")
        s["x"], s["y"] = _train_data(case, seed)
    elif kind == "m0":
        d = _lissajous(case["density"], case["warmup"])
        inst = _grid(case, seed, 8)
        s["n"], S = len(inst), d.samples_per_period
        s["ctx"] = fp.Context(fp.Material(), _drive(d), fp.Tol(), 8)
        s["inst"] = fp.instances_to_device(inst, DEV)
        s["m"], s["dm"] = _empty(s["n"], S, 3), _empty(s["n"], S, 3)
        s["ph"] = _empty(s["n"], 2, case["k_max"] + 1, 2)
    elif kind == "m1":
        s["phi"], s["S"] = _m1_data(case, seed)
        Q, C, K1 = case["Q"], case["C"], case["K1"]
        s["a"], s["eps"], s["smax"] = _empty(Q, C, K1, 2), _empty(Q, C, K1), _empty(C, K1)
        s["ks"], s["ef"], s["eg"] = _ks(case), _empty(K1), _empty(1)
    else:
        s["phi"], s["a"], s["S"], s["smax"] = _m2_data(case, seed)
        s["ks"], s["G"] = _ks(case), _empty(case["J"] + 1, case["J"] + 1, 2)
    return s


# -------------------------------------------------------------------- pass --
def run(s):
    kind = s["kind"]
    if kind == "solve":
        fp.fp_solve_batch(s["ctx"], s["inst"], s["n"], s["m"], s["dm"], s["st"])
        return {"m": s["m"], "dmdt": s["dm"], "status": s["st"]}
    if kind == "sysmat":
        fp.fp_solve_batch(s["ctx"], s["inst"], s["n"], None, s["dm"], s["st"])
        fp.fp_signal(s["ctx"], s["dm"], s["n"], s["k_max"], CH, s["ph"])
        return {"dmdt": s["dm"], "phi_hat": s["ph"], "status": s["st"]}
    if kind == "sweep":
        st = s["stream"]
        st.wait_stream(torch.cuda.current_stream())
        s["sw"].run(s["inst"], s["m"], s["dm"], s["st"], stream=st)
        torch.cuda.current_stream().wait_stream(st)
        return {"m": s["m"], "dmdt": s["dm"], "status": s["st"]}
    if kind == "grad":
        p = s["params"].detach().requires_grad_()
        ph = fp.phi_hat(p, s["h_off"], s["ctx"], s["L"], s["k_max"], CH)
        J = (ph - s["u"]).square().sum()
        J.backward()
        return {"J": J.detach(), "phi_hat": ph.detach(), "grad": p.grad}
    if kind == "ensemble":
        mean, spread = s["net"].infer(s["x"])
        return {"mean": mean, "spread": spread}
    if kind == "infer":
        return {"y": s["net"].infer(s["x"])}
    if kind == "train":
        net = s["net"]
        loss = net.grad(s["x"], s["y"])
        net.adam(1e-3)
        return {"loss": loss, "gW": net.gW, "gb": net.gb, "W": net.Wm, "b": net.bm}
    if kind == "m0":
        fp.fp_equilibrium(s["ctx"], s["inst"], s["n"], s["m"], s["dm"])
        fp.fp_signal(s["ctx"], s["dm"], s["n"], s["k_max"], CH, s["ph"])
        return {"m": s["m"], "dmdt": s["dm"], "phi_hat": s["ph"]}
    if kind == "m1":
        fp.fp_m1_fit(s["phi"], s["Q"], s["S"], s["N"], s["C"], s["K1"], s["a"], s["eps"], s["smax"])
        fp.fp_nrmse(s["eps"], s["Q"], s["C"], s["K1"], s["ks"], len(s["ks"]), s["ef"], s["eg"])
        return {"a": s["a"], "eps": s["eps"], "smax": s["smax"], "eps_freq": s["ef"], "eps_global": s["eg"]}
    fp.fp_m2_gram(s["phi"], s["a"], s["S"], s["smax"], s["A"], s["J"], s["N"], s["C"], s["K1"], s["ks"],
                  len(s["ks"]), s["G"])
    return {"gram": torch.triu(_cplx(s["G"]))}                             # the triangle that the call fills


# -------------------------------------------------------------------- work --
def _solver_flops(n, intervals, L, stages):
    # one step per sample interval, two Newton iterations of stage operator applies (about 17 couplings a row)
    # and stage combinations
    N = (L + 1) ** 2
    return 2.0 * n * intervals * (2 * stages * 17 * N + 2 * N * (2 * stages ** 2 + 3 * stages))


def work(case):
    kind = case["kind"]
    if kind == "solve":
        n, S = case["n"], case["samples"]
        return {"bytes": n * (68 + 48 * S), "flops": _solver_flops(n, S, case["L_max"], case["stages"])}
    if kind in ("sysmat", "m0"):
        n, S = case["nx"] * case["ny"], 102 * case["density"]
        k1 = (case.get("k_max") or S // 2) + 1
        dft = 2 * n * 2.5 * S * math.log2(S)                               # two real transforms
        if kind == "m0":
            return {"bytes": n * (64 + 48 * S + 32 * k1), "flops": dft + 100.0 * n * S}
        return {"bytes": n * (68 + 24 * S + 32 * k1),
                "flops": dft + _solver_flops(n, S * (1 + case["warmup"]), case["L"], case["stages"])}
    if kind == "sweep":
        n, S = case["n"], 102 * case["density"]
        return {"bytes": n * (68 + 48 * S), "flops": _solver_flops(n, S, case["L_max"] - 1, 3)}
    if kind == "grad":
        n, S = case["sets"] * case["nx"] * case["ny"], 102 * case["density"]
        return {"bytes": n * (64 + 32 + 64 * (case["k_max"] + 1)), "flops": 3 * _solver_flops(n, S, case["L"], 3)}
    if kind in ("ensemble", "infer", "train"):
        q, nets = case["q"], 2 if kind == "ensemble" else 1
        mac = 7 * 512 + 3 * 512 * 512 + 512 * 800
        if kind == "train":
            return {"bytes": q * (28 + 3200) + 28.0 * mac, "flops": 6.0 * q * mac}
        return {"bytes": q * (28 + 3200) + nets * 2.0 * mac, "flops": 2.0 * q * mac * nets}
    if kind == "m1":
        e = case["Q"] * case["N"] * case["C"] * case["K1"]
        return {"bytes": 16.0 * (e + case["N"] * case["C"] * case["K1"]) + 24.0 * case["Q"] * case["C"] * case["K1"],
                "flops": 24.0 * e}
    rows = case["A"] * case["N"] * case["C"] * len(_ks_host(case))
    return {"bytes": 16.0 * rows * (case["J"] + 1), "flops": 4.0 * rows * (case["J"] + 1) * (case["J"] + 2)}


def _ks_host(case):
    return fp.fp_freq_index_set(case["orders"], case["orders"], 16, case["K1"] - 1)


# ------------------------------------------------- the same in plain 64 bits --
def _net64(path):
    z = np.load(path)
    W = [torch.from_numpy(z["W%d" % l]).view(torch.bfloat16).double().to(DEV) for l in range(5)]
    W[0] = W[0][:, :7]
    b = [torch.from_numpy(z["b%d" % l]).double().to(DEV) for l in range(5)]
    return W, b, [torch.from_numpy(z[k]).double().to(DEV) for k in ("in_shift", "in_scale", "out_shift", "out_scale")]


def _forward64(net, x):
    W, b, (ish, isc, osh, osc) = net
    h = (x.double() - ish) * isc
    for l in range(4):
        h = torch.nn.functional.gelu(h @ W[l].T + b[l])
    z = h @ W[4].T + b[4]
    return z, z * osc + osh


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        x = _queries(case, seed)
        a, b = _net64(DATA + ".m0.npz"), _net64(DATA + ".m1.npz")
        mean, spread = [], []
        for c in x.split(65536):
            y0, y1 = _forward64(a, c)[1], _forward64(b, c)[1]
            mean.append((y0 + y1) / 2)
            spread.append((y0 - y1).norm(dim=1) / (2 * mean[-1].norm(dim=1)))
        return {"mean": torch.cat(mean), "spread": torch.cat(spread)}
    if kind == "infer":
        net = _net64(DATA + ".m0.npz")
        return {"y": torch.cat([_forward64(net, c)[1] for c in _queries(case, seed).split(65536)])}
    if kind == "train":
        x, y = _train_data(case, seed)
        W, b, norm = _net64(DATA + ".m0.npz")
        W, b = [w.requires_grad_() for w in W], [v.requires_grad_() for v in b]
        z, _ = _forward64((W, b, norm), x)
        loss = (z - (y.double() - norm[2]) / norm[3]).square().sum()
        (loss / (case["q"] * 800)).backward()
        g0 = torch.zeros((512, 64), dtype=torch.float64, device=DEV)
        g0[:, :7] = W[0].grad
        return {"loss": loss.detach().reshape(1), "gW": [g0] + [w.grad for w in W[1:]], "gb": [v.grad for v in b],
                "W": None, "b": None}
    if kind == "m0":
        d = _lissajous(case["density"], case["warmup"])
        inst = _grid(case, seed, 8)
        S = d.samples_per_period
        t = (d.warmup_periods + torch.arange(S, dtype=torch.float64, device=DEV) / S) * d.period
        off = torch.from_numpy(np.ascontiguousarray(inst["h_off"])).to(DEV)
        w = 2 * np.pi * torch.tensor(d.freq, dtype=torch.float64, device=DEV)
        amp, ph = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (d.amp, d.phase))
        arg = t[:, None] * w + ph
        B = off[:, None, :] + amp * torch.sin(arg)
        Bd = (amp * w * torch.cos(arg))[None]
        dia = float(inst["d"][0])
        bT = np.pi * dia ** 3 / 6.0 * 474e3 / (KB * 293.0)
        nb = B.norm(dim=-1, keepdim=True).clamp_min(1e-300)
        x = bT * nb
        small = x < 0.3
        xs = torch.where(small, torch.ones_like(x), x)
        x2 = torch.where(small, x, torch.zeros_like(x)) ** 2
        c = [1 / 3, -1 / 45, 2 / 945, -1 / 4725, 2 / 93555, -1382 / 638512875, 4 / 18243225, -3617 / 162820783125]
        g = torch.where(small, sum(c[k] * x2 ** k for k in range(8)), (1 / torch.tanh(xs) - 1 / xs) / xs)     # L / x
        dL = torch.where(small, sum((2 * k + 1) * c[k] * x2 ** k for k in range(8)), 1 / xs ** 2 - 1 / torch.sinh(xs) ** 2)
        e = B / nb
        m = bT * g * B
        dm = bT * (g * Bd + (dL - g) * (e * Bd).sum(-1, keepdim=True) * e)
        u = torch.fft.fft(dm[..., :2].transpose(1, 2), dim=-1) / S
        return {"m": m, "dmdt": dm, "phi_hat": torch.view_as_real(u[..., :case["k_max"] + 1].contiguous())}
    if kind == "m1":
        phi, S = _m1_data(case, seed)
        Sc = _cplx(S)
        smax = Sc.abs().amax(0)
        a, eps = [], []
        for q in range(case["Q"]):
            p = _cplx(phi[q])
            a.append((Sc * p.conj()).sum(0) / p.abs().square().sum(0))
            eps.append((Sc - a[-1] * p).abs().square().mean(0).sqrt() / smax)
        a, eps = torch.stack(a), torch.stack(eps)
        ef2 = eps.square().mean(dim=(0, 1))
        return {"a": torch.view_as_real(a), "eps": eps, "smax": smax, "eps_freq": ef2.sqrt(),
                "eps_global": ef2[_ks(case).long()].mean().sqrt().reshape(1)}
    if kind == "m2":
        phi, a, S, smax = _m2_data(case, seed)
        k = _ks(case).long()
        G = 0
        for t in range(case["A"]):
            M = (_cplx(a[t])[:, None] * _cplx(phi[t]))[..., k]             # [J, N, C, k]
            M = torch.cat([M, _cplx(S[t])[None][..., k]]) / smax[t][..., k]
            M = M.reshape(case["J"] + 1, -1)
            G = G + M.conj() @ M.T
        return {"gram": torch.triu(G)}
    return None                                                            # an adaptive integration has no short form
