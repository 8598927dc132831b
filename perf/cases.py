"""The work a user of this library has it do, as cases to time.

Every case is one call (or one call and the read of its spectrum) through the public Python entry
points of ``paper_2602_13198_gb300.mc``.  The sizes are those of the configurations, the tests and the
benchmark of this repository, or shares of them that one pass finishes well within two seconds:

* the per-zone emission counts alone (planning a job, device tensors in and out);
* the flat and Schwarzschild synchrotron spheres, with and without Compton scattering;
* the 2-D torus and the turbulent 3-D snapshot (one shard of the job, as a rank of a sharded job runs it);
* the batched parameter survey;

in every precision form (FP64, mixed, split), with the coefficient network, and with kappa electrons
and bremsstrahlung.  The fluid's perturbations and the Philox seed come from the case's seed.
"""
import math

import numpy as np
import torch

from paper_2602_13198_gb300 import mc, synth

# ------------------------------------------------------------------------------------------ cases
# family, precision form, grid (n1, n2, n3), N_s target, shards of the job (one is run)


def listed():
    return [
        # Emission counts of a 2-D snapshot into the caller's tensors: what a program calls to size a job.
        dict(name="counts_torus2d", kind="counts", n1=256, n2=128, n3=1, n_s=1e6),
        # The smoke run's sphere: the smallest job, bounded by launches and by one path's latency.
        dict(name="sphere_small_fp64", kind="scatter_sphere", prec="fp64", n1=64, n2=32, n3=1, n_s=2e3, tau=0.1),
        # Section 4.1's thin flat sphere at its N_s = 1e5, the spectrum that is compared with theory.
        dict(name="thin_sphere_fp64", kind="thin_sphere", prec="fp64", n1=1024, n2=128, n3=1, n_s=1e5),
        # Scattering sphere of section 4.2 in FP64 (1024 x 128).
        dict(name="scatter_sphere_fp64", kind="scatter_sphere", prec="fp64", n1=1024, n2=128, n3=1, n_s=1e6, tau=0.01),
        # The same in the mixed form, at the largest Thomson depth.
        dict(name="scatter_sphere_mixed", kind="scatter_sphere", prec="mixed", n1=1024, n2=128, n3=1, n_s=3e6, tau=0.1),
        # 2-D torus snapshot (256 x 128, a = 0.9375), plain FP64.
        dict(name="torus2d_fp64", kind="torus", prec="fp64", a=0.9375, n1=256, n2=128, n3=1, n_s=2e6),
        # The same snapshot in the mixed form with the coefficient network.
        dict(name="torus2d_mixed_net", kind="torus", prec="mixed", net=True, a=0.9375, n1=256, n2=128, n3=1, n_s=2e6),
        # kappa electrons and bremsstrahlung on a small ragged retrograde torus, split form.
        dict(name="torus_kappa_brems_split", kind="torus", prec="split", a=-0.94, n1=97, n2=49, n3=1, n_s=3e5,
             kappa=4.5, brems=1, r_high=1.0),
        # One shard of the 3-D snapshot job (288 x 128 x 128 FP32 fields, 6 inclination bins), plain FP64:
        # the benchmark's workload.
        dict(name="snapshot3d_fp64", kind="torus", prec="fp64", a=0.5, n1=288, n2=128, n3=128, n_s=1e8, shards=16),
        # The same shard in the mixed form.
        dict(name="snapshot3d_mixed", kind="torus", prec="mixed", a=0.5, n1=288, n2=128, n3=128, n_s=1e8, shards=16),
        # The same shard in the configuration's stated form: FP64 geodesic, FP32 rest, network.
        dict(name="snapshot3d_split_net", kind="torus", prec="split", net=True, a=0.5, n1=288, n2=128, n3=128, n_s=1e8,
             shards=16),
        # Parameter survey (spin x R_high x accretion rate, uneven grids and N_s) in one batched launch.
        dict(name="survey_mixed", kind="survey", prec="mixed", models=16, n_s=3e5),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["counts", "thin_sphere", "scatter_sphere", "torus", "torus", "torus3d", "torus3d", "survey"])
    prec = rng.choice(["fp64", "mixed", "split"])
    spin = rng.choice([-0.94, -0.5, 0.0, 0.5, 0.9375])
    if kind == "counts":
        return dict(kind="counts", n1=int(_logu(rng, 48, 512)), n2=int(_logu(rng, 24, 200)), n3=1,
                    n_s=_logu(rng, 1e3, 1e8))
    if kind == "thin_sphere":
        return dict(kind=kind, prec=prec, n1=int(_logu(rng, 64, 2048)), n2=int(_logu(rng, 16, 128)), n3=1,
                    n_s=_logu(rng, 1e3, 1e6))
    if kind == "scatter_sphere":
        return dict(kind=kind, prec=prec, n1=int(_logu(rng, 64, 1024)), n2=int(_logu(rng, 32, 128)), n3=1,
                    n_s=_logu(rng, 1e3, 2e6), tau=rng.choice([1e-4, 1e-3, 1e-2, 1e-1]))
    if kind == "survey":
        return dict(kind=kind, prec=prec, models=rng.randint(2, 16), n_s=_logu(rng, 2e4, 3e5))
    net = prec != "fp64" and rng.random() < 0.3
    kappa, brems = 0.0, 0
    if not net and rng.random() < 0.25:
        kappa, brems = rng.choice([(3.5, 0), (5.0, 1), (0.0, 1)])
    if kind == "torus3d":
        n1, n2, n3 = int(_logu(rng, 64, 256)), int(_logu(rng, 32, 128)), int(_logu(rng, 8, 128))
    else:
        n1, n2, n3 = int(_logu(rng, 96, 288)), int(_logu(rng, 48, 160)), 1
    r_high = rng.choice([1.0, 10.0, 20.0])   # hotter electrons: more of the N_s emitted, more scatterings each
    return dict(kind="torus", prec=prec, net=net, a=spin, n1=n1, n2=n2, n3=n3,
                n_s=_logu(rng, 1e4, 2e6 if r_high == 20.0 else 4e5), kappa=kappa, brems=brems, r_high=r_high)


# ----------------------------------------------------------------------------------------- inputs
_BASE = {}


def _torus_base(a, n1, n2, r_high, m_unit):
    """Unperturbed axisymmetric torus (set-up on the host, once per shape): (params, grid), both to be copied."""
    key = (a, n1, n2, r_high, m_unit)
    if key not in _BASE:
        if len(_BASE) > 64:
            _BASE.clear()
        _BASE[key] = synth.torus(a=a, n1=n1, n2=n2, pert=0.0, R_high=r_high, M_unit=m_unit)
    p, g = _BASE[key]
    return dict(p), dict(g)


def _perturbed(g, n3, gen, dtype):
    """Primitives [8, nz] on the GPU: 10% lognormal zone noise on rho and u; on 3-D grids also one
    lognormal turbulent field with P(k) ~ k^-11/3 and standard deviation 0.1."""
    n1, n2 = g["n1"], g["n2"]
    base = torch.as_tensor(g["prim"], device="cuda", dtype=torch.float64).reshape(8, n1, n2, 1)
    prim = base.expand(8, n1, n2, n3).clone()

    def noise():
        return torch.randn((n1, n2, n3), generator=gen, device="cuda", dtype=torch.float64)

    for f in (0, 1):
        prim[f] *= torch.exp(0.1 * noise() - 0.005)
    if n3 > 1:
        k = [torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) for n in (n1, n2, n3)]
        k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
        k2[0, 0, 0] = 1.0
        amp = k2 ** (-11.0 / 12.0)
        amp[0, 0, 0] = 0.0
        d = torch.fft.ifftn(torch.fft.fftn(noise()) * amp).real
        d *= 0.1 / d.std()
        prim[:2] *= torch.exp(d - 0.005)
    return prim.reshape(8, -1).to(dtype).contiguous()


_NET = []


def _network():
    """Weights of the coefficient network: seeded hidden layers and an output layer fitted to the three
    target functions by least squares (rounded to 2^-10), as any program keeps trained weights."""
    if _NET:
        return _NET[0]
    rng = np.random.default_rng(7)
    w1, b1 = rng.normal(0, 1.2, (64, 3)), rng.normal(0, 0.6, 64)
    w2, b2 = rng.normal(0, 0.25, (64, 64)), rng.normal(0, 0.3, 64)
    q = lambda v: np.round(v * 1024.0) / 1024.0  # noqa: E731
    w1, b1, w2, b2 = q(w1), q(b1), q(w2), q(b2)
    x = rng.uniform(-1, 1, (3000, 3))
    th, kk, ep = np.exp(x[:, 0] * math.log(1e3)), np.exp(x[:, 1] * math.log(1e4)), np.exp(x[:, 2] * math.log(1e9) + math.log(1e-3))
    gx, gw = np.polynomial.legendre.leggauss(24)
    # hot cross-section: Maxwell-Juettner average of (1 - mu beta) sigma_KN
    s, sw = 4.0 * (gx + 1.0), 4.0 * gw
    gam = 1.0 + th[:, None] * s * s
    wt = sw * gam * s * s * np.sqrt(th[:, None] * (2.0 + th[:, None] * s * s)) * np.exp(-s * s)
    om = 1.0 - np.sqrt(1.0 - 1.0 / gam ** 2)[:, :, None] * gx
    e = np.maximum(ep[:, None, None] * gam[:, :, None] * om, 1e-3)
    kn = 0.75 / e ** 2 * (2 + e * e * (1 + e) / (1 + 2 * e) ** 2 + (e * e - 2 * e - 2) / (2 * e) * np.log1p(2 * e))
    o0 = np.log((wt * (0.5 * gw * om * kn).sum(-1)).sum(-1) / wt.sum(-1))
    # K2(1/Theta) over 2 Theta^2 (Theta >= 0.3) and the angle-averaged emissivity shape
    z = 1.0 / np.maximum(th, 0.3)
    t = np.arange(1, 1500) * 0.008
    k2 = 0.008 * (0.5 * np.exp(-z) + (np.exp(-z[:, None] * np.cosh(t)) * np.cosh(2 * t)).sum(-1))
    o1 = np.log(k2) - np.log(2.0 / z ** 2)
    sn = np.sin(0.25 * math.pi * (gx + 1.0))
    big = kk[:, None] / sn
    o2 = np.log((gw * sn * sn * (big ** 0.5 + 2 ** (11 / 12) * big ** (1 / 6)) ** 2 * np.exp(-big ** (1 / 3))).sum(-1)) / 10.0
    silu = lambda v: v / (1.0 + np.exp(-v))  # noqa: E731
    h = silu(silu(x @ w1.T + b1) @ w2.T + b2)
    hb = np.concatenate([h, np.ones((len(h), 1))], 1)
    sol = np.linalg.solve(hb.T @ hb + 1e-3 * np.eye(65), hb.T @ np.stack([o0, o1, o2], 1))
    w3, b3 = q(sol[:64].T), q(sol[64])
    _NET.append(np.concatenate([v.ravel() for v in (w1, b1, w2, b2, w3, b3)]).astype(np.float32))
    return _NET[0]


def _survey(case, seed, gen):
    """The survey's draw at a smaller scale: models over spin, R_high, accretion rate and grid size, N_s
    log-uniform over a factor of 100 up to the case's n_s."""
    rng = np.random.default_rng(1)   # the survey is the same one; its fluid and photons follow the seed
    out = []
    for i in range(case["models"]):
        a = [-0.94, -0.5, 0.0, 0.5, 0.94][rng.integers(5)]
        rh = [1.0, 10.0, 40.0, 160.0][rng.integers(4)]
        scale = [0.5, 1.0, 2.0, 4.0][rng.integers(4)]
        n1, n2 = [(128, 64), (192, 96), (256, 128)][rng.integers(3)]
        n_s = case["n_s"] * 10.0 ** rng.uniform(-2.0, 0.0)
        p, g = _torus_base(a, n1, n2, rh, 5e17 * scale)
        m = mc.Model(p, device=0, precision=case["prec"])
        m.set_grid(g, prim=_perturbed(g, 1, gen, torch.float64))
        out.append((m, n_s, seed * 1000 + i))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "survey":
        models = _survey(case, seed, gen)
        return dict(kind=kind, models=[m for m, _, _ in models], n_s=[n for _, n, _ in models],
                    seeds=[s for _, _, s in models])
    if kind == "thin_sphere":
        p, g = synth.sphere("flat", R=1.0, ne=1e13, thetae=100.0, B_gauss=1.0, n1=case["n1"], n2=case["n2"],
                            r_record=3000.0)
        prim = None
    elif kind == "scatter_sphere":
        p, g = synth.scattering_sphere(case["tau"], n1=case["n1"], n2=case["n2"])
        prim = None
    else:   # torus, and the counts of one
        p, g = _torus_base(case.get("a", 0.9375), case["n1"], case["n2"], case.get("r_high", 20.0), 1e18)
        n3 = case["n3"]
        prim = _perturbed(g, n3, gen, torch.float32 if n3 > 1 else torch.float64)
        g["n3"], g["dx3"] = n3, 2.0 * math.pi / n3
        p.update(kappa=case.get("kappa", 0.0), brems=case.get("brems", 0), n_incl=6 if n3 > 1 else 1)
    m = mc.Model(p, device=0, precision=case.get("prec", "fp64"), surrogate=bool(case.get("net")))
    m.set_grid(g, prim=prim)
    if case.get("net"):
        m.surrogate_weights(_network())
    state = dict(kind=kind, model=m, n_s=float(case["n_s"]), seed=seed, shards=case.get("shards", 1))
    if kind == "counts":
        state["out"] = [torch.empty(n, dtype=torch.int64, device="cuda") for n in (m.nz, m.nz, 1)]
    return state


# -------------------------------------------------------------------------------------------- run
_COUNTERS = ("n_emit", "n_child", "n_rec", "n_abs", "n_capt", "n_maxst", "n_steps", "n_events", "n_total")


def _spectrum(m):
    nu_l, sigma, counts = m.spectrum()
    return dict(nuL=nu_l, sigma=sigma, counts=counts)


def run(state):
    if state["kind"] == "counts":
        counts, start, total = state["out"]
        state["model"].zone_counts_noalloc(state["n_s"], state["seed"], counts, start, total)
        return dict(counts=counts, start=start, total=total)
    if state["kind"] == "survey":
        st = mc.run_batch(state["models"], state["n_s"], state["seeds"])
        out = [_spectrum(m) for m in state["models"]]
        both = {k: np.stack([o[k] for o in out]) for k in out[0]}
    else:
        m = state["model"]
        st = m.run(state["n_s"], state["seed"], shard=0, n_shards=state["shards"])
        both = _spectrum(m)
    both["stats"] = np.array([st[k] for k in _COUNTERS], dtype=np.int64)
    return both


# ------------------------------------------------------------------------------------------- work
# Per family, measured: primaries per N_s, superphotons (with their scattered descendants) per primary,
# geodesic steps per superphoton, share of the steps inside the grid.
_FAMILY = {
    "thin_sphere": (0.84, 1.0, 290.0, 0.21),
    "scatter_sphere": (0.79, 1.03, 95.0, 0.36),
    "torus": (0.3, 2.5, 193.0, 0.54),
    "torus_hot": (1.0, 3.8, 183.0, 0.44),
    "torus3d": (0.225, 1.43, 203.0, 0.565),
    "survey": (0.21, 2.85, 184.0, 0.5),
}


def work(case):
    zones = case.get("n1", 192) * case.get("n2", 96) * case.get("n3", 1) * case.get("models", 1)
    size = 4 if case.get("n3", 1) > 1 else 8
    # one emissivity per zone and frequency node (200), about 30 operations each
    flops, nbytes = zones * 200 * 30.0, zones * 8.0 * size
    if case["kind"] == "counts":
        return dict(bytes=nbytes + 16.0 * zones, flops=flops)
    family = case["kind"]
    if family == "torus" and case.get("r_high", 20.0) < 20.0:
        family = "torus_hot"
    elif family == "torus" and case["n3"] > 1:
        family = "torus3d"
    prim, per, steps, inside = _FAMILY[family]
    n = case["n_s"] * prim * per / case.get("shards", 1)
    if case["kind"] == "survey":
        n *= case["models"] * 0.31   # the mean of the survey's N_s over their largest
    # operations of one step: geodesic 276, and inside the grid the plasma state and coefficients 340
    flops += n * (2000.0 + steps * (276.0 + inside * 340.0))
    bins = 200 * (6 if case.get("n3", 1) > 1 else 1) * case.get("models", 1)
    return dict(bytes=nbytes + 24.0 * bins, flops=flops)


def exact(case, seed):
    """The spectra are Monte Carlo results of some 10^8 dependent random draws: none in 64 bits without the
    method itself within the time, and the counts are whole numbers."""
    return None
