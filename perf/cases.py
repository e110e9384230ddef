"""The performance cases of the framework: what a user's program asks of it, from one template of
a likelihood step to the full survey estimate, each through the public entry points of
``paper_2202_11839_gb300.lpp``.

Kinds of case
  estimate   Plan.assign + Plan.multipoles: all requested multipoles of one catalogue
  batch      Batch.launch + Batch.results: several mocks on mixed grids in one CUDA graph
  window     Plan.assign + Plan.window_q: Q_l(s) of the randoms by FFT correlations
  pairs      window_q_pairs: Q_l(s) by FP64 pair counts
  template   Template.derived / Template(...): window-convolved theory templates
  predict    Surrogate.predict: emulated curves
  train      Surrogate.train: a schedule of Adam steps, and the updated weights

Inputs are drawn on the device from the seed: a Gaussian density field with a BBKS spectrum and its
tidal tensor, galaxies thinned by 1 + delta, shapes -T_ij plus Gaussian shape noise.  ``exact``
restates every path in 64 bits with plain torch and numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_11839_gb300 import lpp as L

POLE = (-1.0, 0.0, 0.0)
OBSERVER_DISTANCE = 4000.0      # periodic boxes: the observer sits this far below the centre
ALL = L.LPP_WANT_ALL
MOMENTS = {"all": ALL, "all+b": ALL | L.LPP_WANT_CROSS_B, "all+density": ALL | L.LPP_WANT_DENSITY}
# parameter box of the templates: A, b_g, sigma_8, tilt, Gamma, shot-noise scale
RANGES = np.array([[0.0, 3.0], [1.0, 3.0], [0.6, 1.0], [-0.2, 0.2], [0.1, 0.3], [0.5, 2.0]])
FEED = (0, 0, 0, 1, 1, 0)
NODES = 8
SIZES = (6, 256, 256, 256, 256, 320)


# ------------------------------------------------------------------------------- the cases
def _estimate(name, n, count, *, geometry="box", box=2000.0, randoms=0, tsc=True, interlace=True, fp64=False,
              gamma=False, weights=False, host=False, kfrac=0.995, bins=40, moments="all"):
    return {"name": name, "kind": "estimate", "n": n, "count": count, "geometry": geometry, "box": box,
            "randoms": randoms, "tsc": tsc, "interlace": interlace, "fp64": fp64, "gamma": gamma,
            "weights": weights, "host": host, "kfrac": kfrac, "bins": bins, "moments": moments}


def listed():
    return [
        # the headline workload: a polar-cap survey on 512^3, 1.5M shapes and 15M randoms, k to half of Nyquist
        _estimate("survey_512", 512, 1_500_000, geometry="survey", box=4000.0, randoms=15_000_000, kfrac=0.4974),
        # one realisation of the periodic validation mocks (periodic_L2000_N256_tsc_il.json)
        _estimate("periodic_256", 256, 2_000_000),
        # the FP64 reference plan (periodic_L500_N64_cic_fp64.json): precision studies and tests
        _estimate("periodic_64_f64", 64, 50_000, box=500.0, tsc=False, interlace=False, fp64=True, kfrac=1.0,
                  bins=20),
        # a quick look at a small catalogue held in numpy: measured ellipticities and weights, an odd count,
        # the host-to-device copies inside the call
        _estimate("quicklook_64", 64, 20_011, gamma=True, weights=True, host=True, bins=20, kfrac=0.8),
        # a covariance run: small mocks on mixed grids through one captured graph
        {"name": "batch_8", "kind": "batch", "mocks": 8, "n0": 64, "n1": 128, "low": 60_000, "high": 250_000},
        # window multipoles of a survey's randoms on its padded grid
        {"name": "window_256", "kind": "window", "n": 256, "count": 1_000_003, "bins": 100, "fp64": False},
        # the pair-count cross-check of the window on a subsample
        {"name": "pairs_20k", "kind": "pairs", "count": 20_001, "bins": 40, "box": 0.0},
        # training and test sets of the emulator: derived curves of thousands of parameter sets
        {"name": "templates_8192", "kind": "template", "count": 8192, "bins": 40, "derived": True, "png": False},
        # one likelihood evaluation of a chain: all native slots of one parameter set
        {"name": "template_1", "kind": "template", "count": 1, "bins": 40, "derived": False, "png": False},
        # the emulator in bulk, and for the walkers of one ensemble step
        {"name": "predict_8192", "kind": "predict", "count": 8192, "chunk": 8192},
        {"name": "predict_50", "kind": "predict", "count": 50, "chunk": 256},
        # part of one learning-rate phase at the default minibatch
        {"name": "train_256", "kind": "train", "batch": 256, "steps": 200, "rows": 20_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estimate", "estimate", "estimate", "estimate", "batch", "window", "pairs", "template",
                       "predict", "train"])
    if kind == "estimate":
        n = rng.choice([32, 64, 64, 128, 128, 256, 256, 512])
        if n == 512:
            c = _estimate("", n, _log(rng, 100_000, 1_400_000), geometry="survey", box=4000.0,
                          randoms=_log(rng, 1_000_000, 10_000_000), kfrac=rng.uniform(0.3, 0.49))
        else:
            survey = rng.random() < 0.4
            count = _log(rng, 2_000, min(2_000_000, n ** 3 // 4))
            c = _estimate("", n, count, geometry="survey" if survey else "box",
                          box=float(rng.choice([1000, 2000, 4000])), randoms=_log(rng, 5, 10) * count if survey else 0,
                          tsc=rng.random() < 0.7, interlace=rng.random() < 0.7, fp64=n <= 64 and rng.random() < 0.4,
                          gamma=rng.random() < 0.4, weights=rng.random() < 0.5, host=rng.random() < 0.25,
                          kfrac=round(rng.uniform(0.4, 0.995), 3), bins=rng.randint(10, 50),
                          moments=rng.choice(["all", "all", "all+b", "all+density"]) if n <= 128 else "all")
    elif kind == "batch":
        n0 = rng.choice([32, 64, 128])
        c = {"kind": kind, "mocks": rng.randint(2, 12), "n0": n0, "n1": min(128, 2 * n0), "low": n0 ** 3 // 16,
             "high": n0 ** 3 // 4 + rng.randint(1, 9999)}
    elif kind == "window":
        c = {"kind": kind, "n": rng.choice([64, 128, 256]), "count": _log(rng, 20_000, 1_000_000),
             "bins": rng.randint(20, 150), "fp64": False}
        c["fp64"] = c["n"] <= 64 and rng.random() < 0.5
    elif kind == "pairs":
        c = {"kind": kind, "count": _log(rng, 1_000, 20_000), "bins": rng.randint(10, 60),
             "box": rng.choice([0.0, 1000.0])}
    elif kind == "template":
        c = {"kind": kind, "count": _log(rng, 1, 8000), "bins": rng.randint(15, 60), "derived": rng.random() < 0.5,
             "png": rng.random() < 0.25}
    elif kind == "predict":
        c = {"kind": kind, "count": _log(rng, 1, 8192), "chunk": rng.choice([256, 1024, 8192])}
    else:
        c = {"kind": kind, "batch": rng.choice([64, 96, 128, 256, 512]), "steps": rng.randint(40, 190),
             "rows": _log(rng, 2_000, 20_000)}
    return {k: v for k, v in c.items() if k != "name"}


def _fields(moments):
    return 136 + (27 if moments == "all+b" else 14 if moments == "all+density" else 0)


def work(case):
    """Each input read once and each output written once; the transforms, the assignment and the
    per-mode products that the estimator is defined by, without its present intermediate grids."""
    k = case["kind"]
    if k in ("estimate", "batch"):
        es = 8 if case.get("fp64") else 4
        if k == "estimate":
            jobs = [(case["n"], case["count"], case["randoms"], case["interlace"], _fields(case["moments"]))]
        else:
            mean = (case["low"] + case["high"]) // 2
            jobs = [(case["n0"] if j % 2 == 0 else case["n1"], mean, 0, True, 136) for j in range(case["mocks"])]
        cells = 27 if case.get("tsc", True) else 8
        b = f = 0.0
        for n, count, rand, il, fields in jobs:
            b += count * es * (3 + 1 + (2 if case.get("gamma") else 6)) + rand * es * 5 + 14 * 50 * 16
            f += fields * ((2 if il else 1) * (2.5 * n ** 3 * math.log2(n ** 3) + 2.0 * cells * count) + 8.0 * n ** 3)
        return {"bytes": b, "flops": f}
    if k == "window":
        n, es = case["n"], 8 if case["fp64"] else 4
        return {"bytes": case["count"] * es * 5.0 + 5 * 8 * case["bins"],
                "flops": 46 * 2 * 2.5 * n ** 3 * math.log2(n ** 3) + 46 * 54.0 * case["count"]}
    if k == "pairs":
        return {"bytes": case["count"] * 8 * 5.0, "flops": case["count"] ** 2 / 2 * 60.0}
    if k == "template":
        nt, slots = case["count"], 9 if case["derived"] else 14
        return {"bytes": nt * (48.0 + 14 * case["bins"] * 8 + (32 * case["bins"] if case["derived"] else 0)),
                "flops": nt * (2048 * 60.0 + slots * case["bins"] * 2 * 2048.0)}
    par = sum(a * b + b for a, b in zip(SIZES[:-1], SIZES[1:]))
    if k == "predict":
        return {"bytes": case["count"] * (48.0 + 1280) + 4.0 * par, "flops": case["count"] * (2.0 * par + 2 * 64 * 320)}
    return {"bytes": case["steps"] * case["batch"] * 1304.0 + 8.0 * par, "flops": case["steps"] * case["batch"] * 6.0 * par}


# ------------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _generator(seed, stream=0):
    g = torch.Generator(device=_device())
    g.manual_seed(1_000_003 * int(seed) + 7919 * stream + 17)
    return g


def _density_field(box, g, nf=64):
    """delta and the six tidal components (xx, yy, zz, xy, xz, yz) of a BBKS Gaussian field, nf^3."""
    dev = _device()
    white = torch.randn((nf, nf, nf), generator=g, device=dev, dtype=torch.float64)
    dk = torch.fft.fftn(white)
    f = torch.fft.fftfreq(nf, d=1.0 / nf, device=dev, dtype=torch.float64) * (2.0 * math.pi / box)
    k = torch.meshgrid(f, f, f, indexing="ij")
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    q = torch.sqrt(k2) / 0.2
    t = torch.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    p = q * t * t
    p[0, 0, 0] = 0.0
    dk = dk * torch.sqrt(p)
    delta = torch.fft.ifftn(dk).real
    amp = 0.5 / delta.std()
    tid = [torch.fft.ifftn(dk * (k[i] * k[j] / k2 - (1.0 / 3.0 if i == j else 0.0))).real * amp
           for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    return delta * amp, torch.stack(tid).reshape(6, -1)


def _observer(geometry, box):
    return (box / 2, box / 2, 0.05 * box) if geometry == "survey" else (box / 2, box / 2, box / 2 - OBSERVER_DISTANCE)


def _points(count, geometry, box, g):
    """Uniform points of the box, or of the polar cap theta < 60 deg with n(r) peaked mid-shell."""
    dev = _device()
    if geometry == "box":
        return torch.rand((3, count), generator=g, device=dev, dtype=torch.float64) * box
    lo, hi, mean, sig = 0.25 * box, 0.45 * box, 0.35 * box, 0.05 * box
    out = torch.empty((3, 0), device=dev, dtype=torch.float64)
    while out.shape[1] < count:
        m = int((count - out.shape[1]) * 2.2) + 1024
        r = torch.randn(m, generator=g, device=dev, dtype=torch.float64) * sig + mean
        v = torch.rand((3, m), generator=g, device=dev, dtype=torch.float64)
        mu, ph = 0.5 + 0.5 * v[0], 2 * math.pi * v[1]
        st = torch.sqrt(1 - mu * mu)
        ok = (r > lo) & (r < hi) & (v[2] < (r / hi) ** 2)
        p = torch.stack([r * st * torch.cos(ph), r * st * torch.sin(ph), r * mu])[:, ok]
        out = torch.cat([out, p], dim=1)
    out = out[:, :count]
    return out + torch.tensor(_observer("survey", box), device=dev, dtype=torch.float64)[:, None]


def _inside(pos, box, dtype):
    """Positions in the plan's precision, strictly inside the box after rounding."""
    lim = torch.tensor(box, dtype=dtype)
    return pos.to(dtype).clamp_(min=0.0, max=float(torch.nextafter(lim, torch.zeros_like(lim)))).contiguous()


def _nbar(pos, box, scale):
    obs = torch.tensor(_observer("survey", box), device=pos.device, dtype=pos.dtype)[:, None]
    r = torch.sqrt(((pos - obs) ** 2).sum(0))
    return scale * torch.exp(-0.5 * ((r - 0.35 * box) / (0.05 * box)) ** 2)


def _catalogue(count, geometry, box, seed, dtype, gamma, weights, stream=0):
    """Galaxies thinned by 1 + delta, with shapes -T_ij plus isotropic noise (sigma = 0.25)."""
    g = _generator(seed, stream)
    dev = _device()
    delta, tid = _density_field(box, g)
    nf = delta.shape[0]
    one = (1.0 + delta).clamp_(0.0, 3.0).reshape(-1)
    pos = torch.empty((3, 0), device=dev, dtype=torch.float64)
    while pos.shape[1] < count:
        c = _points(int((count - pos.shape[1]) * 3.2) + 256, geometry, box, g)
        u = torch.rand(c.shape[1], generator=g, device=dev, dtype=torch.float64)
        i = (c / box * nf).long().clamp_(0, nf - 1)
        pos = torch.cat([pos, c[:, u * 3.0 < one[(i[0] * nf + i[1]) * nf + i[2]]]], dim=1)
    pos = pos[:, :count]
    i = (pos / box * nf).long().clamp_(0, nf - 1)
    s = -tid[:, (i[0] * nf + i[1]) * nf + i[2]]
    z = torch.randn((5, count), generator=g, device=dev, dtype=torch.float64) * (math.sqrt(2.0) * 0.25)
    if gamma:
        shape = torch.stack([0.5 * (s[0] - s[1]), s[3]]) + z[:2] / math.sqrt(2.0)
    else:
        r2, r6 = math.sqrt(2.0), math.sqrt(6.0)
        shape = s + torch.stack([z[0] / r2 + z[1] / r6, -z[0] / r2 + z[1] / r6, -2 * z[1] / r6, z[2] / r2, z[3] / r2,
                                 z[4] / r2])
    w = 0.5 + torch.rand(count, generator=g, device=dev, dtype=torch.float64) if weights else None
    return (_inside(pos, box, dtype), None if w is None else w.to(dtype), shape.to(dtype).contiguous())


def _random_points(count, box, seed, dtype, scale, weights=False):
    g = _generator(seed, 101)
    pos = _points(count, "survey", box, g)
    nbar = _nbar(pos, box, scale)
    w = 0.5 + torch.rand(count, generator=g, device=pos.device, dtype=torch.float64) if weights else None
    return _inside(pos, box, dtype), None if w is None else w.to(dtype), nbar.to(dtype)


def _estimate_inputs(case, seed):
    dtype = torch.float64 if case["fp64"] else torch.float32
    pos, w, shape = _catalogue(case["count"], case["geometry"], case["box"], seed, dtype, case["gamma"], case["weights"])
    ran = None
    if case["randoms"]:
        ran = _random_points(case["randoms"], case["box"], seed, dtype, case["count"] / (0.05 * case["box"] ** 3))
    return pos, w, shape, ran


def _edges(n, box, kfrac, bins):
    return np.linspace(0.0, kfrac * math.pi * n / box, bins + 1)


def _batch_inputs(case, seed):
    sizes = np.random.default_rng(seed).integers(case["low"], case["high"] + 1, case["mocks"])
    return [(case["n0"] if j % 2 == 0 else case["n1"],) +
            _catalogue(int(sizes[j]), "box", 1000.0, seed, torch.float32, False, False, stream=j)
            for j in range(case["mocks"])]


def _window_inputs(case, seed):
    return _random_points(case["count"], 2000.0, seed, torch.float64 if case["fp64"] else torch.float32, 1e-3, True)


def _pair_inputs(case, seed):
    if case["box"]:
        g = _generator(seed, 3)
        pos = torch.rand((3, case["count"]), generator=g, device=_device(), dtype=torch.float64) * case["box"]
        return pos, 0.5 + torch.rand(case["count"], generator=g, device=_device(), dtype=torch.float64), None
    return _random_points(case["count"], 4000.0, seed, torch.float64, 1e-3, True)


def _pair_geometry(case):
    if case["box"]:
        return (500.0, 500.0, -1500.0), np.linspace(0.0, 400.0, case["bins"] + 1), 0.1
    return _observer("survey", 4000.0), np.linspace(0.0, 2000.0, case["bins"] + 1), 0.1


def _parameters(count, seed):
    u = torch.rand((count, 6), generator=_generator(seed, 5), device=_device(), dtype=torch.float64)
    r = torch.tensor(RANGES, device=u.device)
    return r[:, 0] + u * (r[:, 1] - r[:, 0])


def _window_table(seed):
    """A smooth window table q[5, 190] over separations to 3800 Mpc/h, slightly different for each seed."""
    s = np.linspace(10.0, 3790.0, 190)
    a = 1.0 + 0.05 * np.random.default_rng(seed).standard_normal(5)
    x = s / 1800.0
    q0 = np.clip(1.0 - 1.1 * x + 0.3 * x ** 3, 0.0, None) * np.exp(-0.4 * a[0] * x)
    q = [q0] + [0.4 / (1 + i) * a[i] * (-1) ** (i + 1) * q0 * (1 - np.exp(-(x * 2) ** 2)) for i in range(1, 5)]
    return np.stack(q), s


def _network(seed):
    r = np.random.default_rng(seed)
    out = []
    for fi, fo in zip(SIZES[:-1], SIZES[1:]):
        lim = 1.0 / math.sqrt(fi)
        out.append((r.uniform(-lim, lim, (fo, fi)).astype(np.float32), r.uniform(-0.1, 0.1, fo).astype(np.float32)))
    return out


def _output_map(seed):
    """mu, sd, shot, sigma [320] and the baseline table [64, 320]: smooth curves of (tilt, Gamma) at the
    Lobatto nodes, in units hundreds of times their error bars, as template curves are."""
    r = np.random.default_rng(seed + 1)
    k = np.tile(np.linspace(0.0025, 0.1975, 40), 8)
    amp = np.repeat(np.array([900.0, -400.0, 500.0, -700.0, 250.0, 30.0, -20.0, 10.0]) * r.uniform(0.8, 1.2, 8), 40)
    node = -np.cos(np.pi * np.arange(NODES) / (NODES - 1))
    base = np.stack([amp * (k / 0.05) ** (0.2 * a) / (1 + (k / (0.04 * (2.0 + b))) ** 1.7) for a in node for b in node])
    sigma = 0.02 * np.abs(amp) + 1.0
    return np.zeros(320), 0.05 * sigma, 0.1 * amp * np.exp(-k / 0.1), sigma, base


def _train_rows(case, seed):
    g = _generator(seed, 9)
    x = torch.rand((case["rows"], 6), generator=g, device=_device()) * 2 - 1
    x[:, [0, 1, 2, 5]] = 0.0
    c = torch.randn((6, 320), generator=g, device=_device())
    t, h = x[:, 3:4], x[:, 4:5]
    y = c[0] * t + c[1] * h + c[2] * t * h + 0.5 * c[3] * torch.sin(3 * t) + 0.5 * c[4] * torch.cos(2 * h) + 0.1 * c[5]
    sched = np.concatenate([np.random.default_rng(seed * 100 + e).permutation(case["rows"])
                            for e in range(1 + case["steps"] * case["batch"] // case["rows"])])
    sched = torch.from_numpy(sched[: case["steps"] * case["batch"]].astype(np.int32)).to(_device())
    return x.contiguous(), y.contiguous(), sched


LR = 1e-4


# ------------------------------------------------------------------------------- the passes
def prepare(case, seed):
    k = case["kind"]
    st = {"case": case}
    if k == "estimate":
        pos, w, shape, ran = _estimate_inputs(case, seed)
        if case["host"]:
            pos, w, shape, ran = _numpy(pos), _numpy(w), _numpy(shape), ran and tuple(_numpy(a) for a in ran)
        st["cat"], st["ran"] = (pos, w, shape), ran
        st["plan"] = L.Plan(case["n"], case["box"], _edges(case["n"], case["box"], case["kfrac"], case["bins"]),
                            observer=_observer(case["geometry"], case["box"]), pole=POLE,
                            scheme=L.LPP_TSC if case["tsc"] else L.LPP_CIC, interlace=case["interlace"],
                            precision=L.LPP_FP64 if case["fp64"] else L.LPP_FP32, moments=MOMENTS[case["moments"]],
                            max_shapes=case["count"], max_randoms=case["randoms"], host_inputs=case["host"])
    elif k == "batch":
        mocks = _batch_inputs(case, seed)
        st["mocks"] = mocks
        st["plans"] = []
        grids = sorted({m[0] for m in mocks})
        for n in grids:
            cap = max(m[1].shape[1] for m in mocks if m[0] == n)
            st["plans"].append(L.Plan(n, 1000.0, _edges(n, 1000.0, 0.8, 20), observer=_observer("box", 1000.0),
                                      pole=POLE, scheme=L.LPP_TSC, interlace=True, max_shapes=cap))
        plan_of = [grids.index(m[0]) for m in mocks]
        shapes = [st["plans"][p].particles(L.LPP_SHAPES, m[1], None, None, m[3], L.LPP_SHAPE_TENSOR6)
                  for p, m in zip(plan_of, mocks)]
        st["batch"] = L.Batch(st["plans"], plan_of, shapes, None, use_graph=True, keep=mocks)
    elif k == "window":
        st["ran"] = _window_inputs(case, seed)
        st["edges"] = np.linspace(0.0, 1800.0, case["bins"] + 1)
        st["plan"] = L.Plan(case["n"], 4000.0, np.linspace(0.0, 0.01, 2), origin=(-1000.0,) * 3,
                            observer=_observer("survey", 2000.0), pole=POLE, scheme=L.LPP_TSC,
                            precision=L.LPP_FP64 if case["fp64"] else L.LPP_FP32, moments=1 << L.LPP_MOM_DD0,
                            max_randoms=case["count"])
    elif k == "pairs":
        st["ran"] = _pair_inputs(case, seed)
    elif k == "template":
        q, s = _window_table(seed)
        st["theta"] = _parameters(case["count"], seed)
        st["t"] = L.Template(q, s, np.linspace(0.0, 0.2, case["bins"] + 1), shot_plus=250.0)
        if case["png"]:
            st["t"].set_png(100.0)
        if case["derived"]:
            st["t"].set_slots(L.TEMPLATE_EB_SLOTS)
            st["sigma"] = torch.linspace(50.0, 500.0, 8 * case["bins"], device=_device(), dtype=torch.float64)
    elif k == "predict":
        st["theta"] = _parameters(case["count"], seed)
        st["net"] = L.Surrogate(L.flatten_params(_network(seed)), batch=case["chunk"])
        mu, sd, shot, sigma, base = (torch.from_numpy(a).to(_device()) for a in _output_map(seed))
        st["net"].set_map(RANGES[:, 0], RANGES[:, 1], FEED, mu, sd, shot, None, sigma, base=base, base_nodes=NODES)
    else:
        st["x"], st["y"], st["schedule"] = _train_rows(case, seed)
        st["net"] = L.Surrogate(L.flatten_params(_network(seed)), batch=case["batch"])
        st["losses"] = torch.zeros(case["steps"], dtype=torch.float64, device=_device())
    return st


def _numpy(t):
    return None if t is None else np.ascontiguousarray(t.cpu().numpy())


def _result(est, fp64):
    """An estimate's outputs in the precision of its plan: an FP32 plan's numbers carry FP32 digits."""
    c, r = (np.complex128, np.float64) if fp64 else (np.complex64, np.float32)
    return {"p": est.p.astype(c), "raw": est.raw.astype(c), "k_mean": est.k_mean, "n_modes": est.n_modes,
            "norms": np.array([est.norm_auto, est.norm_cross, est.norm_dd, est.shot_plus, est.shot_dd, est.alpha], dtype=r)}


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "estimate":
        pos, w, shape = st["cat"]
        plan = st["plan"]
        plan.assign(L.LPP_SHAPES, pos, w, None, shape, L.LPP_SHAPE_GAMMA12 if case["gamma"] else L.LPP_SHAPE_TENSOR6)
        if st["ran"]:
            plan.assign(L.LPP_RANDOMS, *st["ran"])
        return _result(plan.multipoles(), case["fp64"])
    if k == "batch":
        st["batch"].launch()
        return [{m: v for m, v in _result(e, False).items() if m in ("p", "raw", "norms")} for e in st["batch"].results()]
    if k == "window":
        st["plan"].assign(L.LPP_RANDOMS, *st["ran"])
        q, s_mean, points, norm = st["plan"].window_q(st["edges"])
        return {"q": q if case["fp64"] else q.astype(np.float32), "s_mean": s_mean, "points": points, "norm": norm}
    if k == "pairs":
        observer, edges, alpha = _pair_geometry(case)
        return L.window_q_pairs(*st["ran"], observer, edges, alpha=alpha, box=case["box"])
    if k == "template":
        if case["derived"]:
            native, curves = st["t"].derived(st["theta"], sigma=st["sigma"])
            return {"native": native, "curves": curves}
        return {"native": st["t"](st["theta"])}
    if k == "predict":
        return st["net"].predict(st["theta"])
    st["net"].train(st["x"], st["y"], st["schedule"], LR, st["losses"])
    return {"params": st["net"].params(), "losses": st["losses"]}


# ------------------------------------------------------------------------------- 64-bit values
def _harmonics(deg, v):
    """Real orthonormal harmonics Y_{deg,n}(v), n = -deg..deg, of unit vectors v [3, ...]."""
    x, y, z = v
    rows = [None] * (2 * deg + 1)
    cs, sn = torch.ones_like(x), torch.zeros_like(x)
    for m in range(deg + 1):
        prev, cur = torch.zeros_like(z), torch.full_like(z, float(math.prod(range(1, 2 * m, 2))))
        for l in range(m + 1, deg + 1):
            prev, cur = cur, ((2 * l - 1) * z * cur - (l + m - 1) * prev) / (l - m)
        norm = math.sqrt((2 * deg + 1) / (4 * math.pi) * math.factorial(deg - m) / math.factorial(deg + m))
        rows[deg + m] = cur * cs * norm * (math.sqrt(2.0) if m else 1.0)
        if m:
            rows[deg - m] = cur * sn * norm * math.sqrt(2.0)
        cs, sn = cs * x - sn * y, cs * y + sn * x
    return torch.stack(rows)


def _legendre_derivative(deg, m):
    c = np.polynomial.legendre.leg2poly([0.0] * deg + [1.0])
    return np.polynomial.polynomial.polyder(c, m) if m else c


def _sphere_nodes(deg):
    """Directions [3, S] and weights of a rule exact for products of two degree-deg harmonics."""
    z, w = np.polynomial.legendre.leggauss(deg + 1)
    ph = 2 * np.pi * np.arange(2 * deg + 1) / (2 * deg + 1)
    st = np.sqrt(1 - z * z)
    d = np.stack([np.outer(st, np.cos(ph)), np.outer(st, np.sin(ph)), np.outer(z, np.ones_like(ph))]).reshape(3, -1)
    return torch.from_numpy(d).to(_device()), torch.from_numpy(np.repeat(w, 2 * deg + 1) * 2 * np.pi / (2 * deg + 1)).to(_device())


def _frames(los):
    p = torch.tensor(POLE, device=los.device, dtype=los.dtype)[:, None].expand_as(los)
    ep = torch.linalg.cross(p, los, dim=0)
    ep = ep / ep.norm(dim=0)
    return torch.linalg.cross(ep, los, dim=0), ep


def _kernel_coefficients(gamma, los, et, ep, spin, deg):
    """c_n = int gamma (k.et - i k.ep)^spin d^spin P_deg(mu) Y_n(k) dk for every galaxy: [2 deg + 1, N] complex."""
    d, wq = _sphere_nodes(deg)
    tab = _harmonics(deg, d) * wq
    poly = _legendre_derivative(deg, spin)
    out = []
    for c0 in range(0, gamma.numel(), 1 << 17):
        c = slice(c0, c0 + (1 << 17))
        mu = d.T @ los[:, c]
        v = torch.zeros_like(mu)
        for a in poly[::-1]:
            v = v * mu + float(a)
        v = v * torch.complex(d.T @ et[:, c], -(d.T @ ep[:, c])) ** spin
        out.append(gamma[c] * torch.complex(tab @ v.real, tab @ v.imag))
    return torch.cat(out, dim=1)


class _Mesh:
    """Assignment, transform and shell sums of one grid in 64 bits (half of the modes, their mirrors implied)."""

    def __init__(self, n, box, tsc, interlace, edges, origin=0.0):
        dev = _device()
        self.n, self.box, self.order, self.interlace, self.origin = n, box, 3 if tsc else 2, interlace, origin
        kf = 2 * math.pi / box
        r = min(n // 2 - 1, int(edges[-1] / kf) + 1)
        a = torch.arange(-r, r + 1, device=dev)
        fz, fy, fx = (t.reshape(-1) for t in torch.meshgrid(a[r:], a, a, indexing="ij"))
        e = torch.tensor(edges, device=dev)
        k = kf * torch.sqrt((fx * fx + fy * fy + fz * fz).double())
        b = torch.bucketize(k, e, right=True) - 1
        keep = (b >= 0) & (b < len(edges) - 1) & ((fz > 0) | (fy > 0) | ((fy == 0) & (fx > 0))) & ((fz > 0) | (fy >= 0))
        fx, fy, fz, self.bin, self.k = fx[keep], fy[keep], fz[keep], b[keep], k[keep]
        self.m = ((fz % n) * n + fy % n) * n + fx % n
        self.mirror = (((-fz) % n) * n + (-fy) % n) * n + (-fx) % n
        f = torch.stack([fx, fy, fz]).double()
        self.khat = f / f.norm(dim=0)
        self.weight = torch.prod(torch.sinc(f / n), dim=0) ** -self.order
        self.phase = torch.polar(torch.ones_like(self.k), -math.pi / n * f.sum(0))
        self.nb = len(edges) - 1

    def axes(self, pos, shift):
        u = (pos.double() - self.origin) * (self.n / self.box) - shift
        if self.order == 2:
            i = torch.floor(u)
            return [(i + j).long() % self.n for j in (0, 1)], [1 - (u - i), u - i]
        i = torch.floor(u + 0.5)
        d = u - i
        return [(i + j).long() % self.n for j in (-1, 0, 1)], [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]

    def deposit(self, grid, pos, values):
        """Adds values at pos to grid [2, n^3] (the second sub-grid is the half-cell shifted one)."""
        for s in range(2 if self.interlace else 1):
            for c0 in range(0, pos.shape[1], 1 << 22):
                c = slice(c0, c0 + (1 << 22))
                i, w = self.axes(pos[:, c], 0.5 * s)
                for a in range(self.order):
                    for b in range(self.order):
                        for d in range(self.order):
                            grid[s].index_add_(0, (i[a][2] * self.n + i[b][1]) * self.n + i[d][0],
                                               values[c] * w[a][2] * w[b][1] * w[d][0])

    def zeros(self):
        return torch.zeros((2, self.n ** 3), device=_device(), dtype=torch.float64)

    def modes(self, grid):
        z = torch.fft.fftn(torch.complex(grid[0], grid[1]).reshape((self.n,) * 3)).reshape(-1)
        a, b = z[self.m], z[self.mirror].conj()
        f = 0.5 * (a + b)
        if self.interlace:
            f = 0.5 * (f + self.phase * (-0.5j) * (a - b))
        return f * self.weight

    def shells(self, t):
        return torch.stack([torch.bincount(self.bin, v, minlength=self.nb) for v in (t.real, t.imag)]).cpu().numpy()


def _exact_estimate(n, box, tsc, interlace, edges, observer, moments, cat, gamma_in, ran):
    mesh = _Mesh(n, box, tsc, interlace, edges)
    nb = mesh.nb
    pos, w, shape = (None if t is None else t.double() for t in cat)
    w = torch.ones(pos.shape[1], device=pos.device, dtype=torch.float64) if w is None else w
    obs = torch.tensor(observer, device=pos.device, dtype=torch.float64)[:, None]
    los = (pos - obs) / (pos - obs).norm(dim=0)
    et, ep = _frames(los)
    if gamma_in:
        gamma = torch.complex(shape[0], shape[1])
    else:
        t = shape[[0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(3, 3, -1)
        tt, pp, tp = (torch.einsum("ap,abp,bp->p", a, t, b) for a, b in ((et, et), (ep, ep), (et, ep)))
        gamma = torch.complex(0.5 * (tt - pp), tp)
    alpha, norm = 0.0, None
    dens = mesh.zeros()
    mesh.deposit(dens, pos, w)
    shot_dd = float((w * w).sum())
    if ran is not None:
        rpos, rw, rn = (None if t is None else t.double() for t in ran)
        rw = torch.ones(rpos.shape[1], device=pos.device, dtype=torch.float64) if rw is None else rw
        alpha = float(w.sum() / rw.sum())
        mesh.deposit(dens, rpos, -alpha * rw)
        norm = alpha * float((rn * rw * rw).sum())
        shot_dd += alpha ** 2 * float((rw * rw).sum())
        rlos = (rpos - obs) / (rpos - obs).norm(dim=0)
    else:
        norm = float(w.sum()) ** 2 / box ** 3

    def transform(values):
        g = mesh.zeros()
        mesh.deposit(g, pos, values)
        return mesh.modes(g)

    d = mesh.modes(dens)
    del dens
    g1, g2 = transform(w * gamma.real), transform(w * gamma.imag)
    raw = np.zeros((L.LPP_N_MOMENTS, 2, nb))
    count = np.maximum(1, 2 * torch.bincount(mesh.bin, minlength=nb).cpu().numpy())
    # sum over a mode and its mirror, where every real field takes its conjugate
    raw[0] = mesh.shells((2 * d.abs() ** 2).to(d.dtype))
    raw[4] = mesh.shells(((g1 + 1j * g2).abs() ** 2 + (g1.conj() + 1j * g2.conj()).abs() ** 2).to(d.dtype))
    plus = (g1.conj() - 1j * g2.conj(), g1 - 1j * g2)
    minus = (g1.conj() + 1j * g2.conj(), g1 + 1j * g2)
    for slot, spin, deg, (pm, pp) in ((1, 2, 2, (d.conj(), d)), (2, 2, 4, (d.conj(), d)), (3, 2, 6, (d.conj(), d)),
                                      (5, 0, 2, plus), (6, 0, 4, plus), (7, 4, 4, minus), (8, 4, 6, minus),
                                      (9, 4, 8, minus)):
        c = _kernel_coefficients(w * gamma, los, et, ep, spin, deg)
        y = _harmonics(deg, mesh.khat)
        sm = torch.zeros_like(d)
        sp = torch.zeros_like(d)
        imag = slot > 3 or moments == "all+b"
        for j in range(2 * deg + 1):
            f = transform(c[j].real.contiguous())
            sm += y[j] * f
            sp += y[j] * f.conj()
            if imag:
                f = transform(c[j].imag.contiguous())
                sm += 1j * y[j] * f
                sp += 1j * y[j] * f.conj()
        raw[slot] = mesh.shells(sm * pm + sp * pp)
        raw[slot] *= (2 * deg + 1) * math.factorial(deg - spin) / math.factorial(deg + spin)
    if moments == "all+density":
        for slot, deg in ((10, 2), (11, 4)):
            y = _harmonics(deg, mesh.khat)
            ys = _harmonics(deg, los)
            yr = None if ran is None else _harmonics(deg, rlos)
            sm = torch.zeros_like(d)
            for j in range(2 * deg + 1):
                g = mesh.zeros()
                mesh.deposit(g, pos, w * ys[j])
                if ran is not None:
                    mesh.deposit(g, rpos, -alpha * rw * yr[j])
                sm += y[j] * mesh.modes(g)
            raw[slot] = 4 * math.pi * mesh.shells(sm * d.conj() + sm.conj() * d)
    raw /= count
    p = raw / norm
    shot_plus = float((w * w * gamma.abs() ** 2).sum()) / norm
    some = torch.bincount(mesh.bin, minlength=nb).cpu().numpy() > 0
    p[0, 0] -= some * shot_dd / norm
    p[4, 0] -= some * shot_plus
    kbar = torch.bincount(mesh.bin, 2 * mesh.k, minlength=nb).cpu().numpy() / count
    return {"p": p[:, 0] + 1j * p[:, 1], "raw": raw[:, 0] + 1j * raw[:, 1], "k_mean": kbar, "n_modes": None,
            "norms": np.array([norm, norm, norm, shot_plus, shot_dd / norm, alpha])}


def _exact_window(case, seed):
    n, box, lo = case["n"], 4000.0, -1000.0
    pos, w, nbar = (t.double() for t in _window_inputs(case, seed))
    mesh = _Mesh(n, box, True, False, np.linspace(0.0, 0.01, 2), lo)
    dev = pos.device
    f = torch.fft.fftfreq(n, d=1.0 / n, device=dev, dtype=torch.float64)
    sinc = torch.sinc(f / n) ** -3
    comp = sinc[:, None, None] * sinc[None, :, None] * sinc[None, None, :]
    obs = torch.tensor(_observer("survey", 2000.0), device=dev, dtype=torch.float64)[:, None]
    y = [_harmonics(l, (pos - obs) / (pos - obs).norm(dim=0)) for l in (0, 2, 4, 6, 8)]

    def transform(values):
        g = mesh.zeros()
        mesh.deposit(g, pos, values)
        return torch.fft.fftn(g[0].reshape((n,) * 3)) * comp

    wk = transform(w)
    h = box / n
    edges = np.linspace(0.0, 1800.0, case["bins"] + 1)
    z, yy, x = torch.meshgrid(f, f, f, indexing="ij")
    s = h * torch.sqrt(x * x + yy * yy + z * z)
    b = torch.bucketize(s, torch.tensor(edges, device=dev), right=True) - 1
    keep = (s > 0) & (b >= 0) & (b < case["bins"])
    b, s, v = b[keep], s[keep], torch.stack([x[keep], yy[keep], z[keep]])
    v = v / v.norm(dim=0)
    cnt = torch.bincount(b, minlength=case["bins"]).cpu().numpy()
    norm = float((nbar * w * w).sum())
    q = np.zeros((5, case["bins"]))
    for i, l in enumerate((0, 2, 4, 6, 8)):
        yk = _harmonics(l, v)
        for j in range(2 * l + 1):
            c = torch.fft.ifftn(transform(w * y[i][j]).conj() * wk).real[keep]
            q[i] += torch.bincount(b, yk[j] * c, minlength=case["bins"]).cpu().numpy()
    q *= 4 * math.pi / (h ** 3 * norm) / np.maximum(1, cnt)
    return {"q": q, "s_mean": torch.bincount(b, s, minlength=case["bins"]).cpu().numpy() / np.maximum(1, cnt),
            "points": None, "norm": norm}


def _exact_pairs(case, seed):
    pos, w, nbar = _pair_inputs(case, seed)
    obs, edges, alpha = _pair_geometry(case)
    nb, n = case["bins"], pos.shape[1]
    e = torch.tensor(edges, device=pos.device)
    los = pos - torch.tensor(obs, device=pos.device, dtype=torch.float64)[:, None]
    los = los / los.norm(dim=0)
    q = torch.zeros((5, nb), device=pos.device, dtype=torch.float64)
    poly = [_legendre_derivative(l, 0) for l in (0, 2, 4, 6, 8)]
    for c0 in range(0, n, 512):
        c = slice(c0, c0 + 512)
        d = pos[:, None, :] - pos[:, c, None]
        if case["box"]:
            d = d - case["box"] * torch.round(d / case["box"])
        s = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        b = torch.bucketize(s, e, right=True) - 1
        ok = (s > 0) & (b >= 0) & (b < nb)
        mu2 = ((d * los[:, c, None]).sum(0)[ok] / s[ok]) ** 2
        ww = (w[c, None] * w[None, :])[ok]
        for i, p in enumerate(poly):
            v = torch.zeros_like(mu2)
            for a in p[::-2]:
                v = v * mu2 + float(a)
            q[i] += torch.bincount(b[ok], ww * v, minlength=nb)
    norm = alpha * float(((1.0 if nbar is None else nbar) * w * w).sum())
    vol = 4 * math.pi / 3 * (edges[1:] ** 3 - edges[:-1] ** 3)
    return q.cpu().numpy() * (2 * np.array([0, 2, 4, 6, 8])[:, None] + 1) * alpha ** 2 / (norm * vol)


def _log_gamma(z):
    shift = 0j
    while z.real.min() < 15.0:
        shift = shift - np.log(z)
        z = z + 1.0
    b = (1 / 6, -1 / 30, 1 / 42, -1 / 30, 5 / 66, -691 / 2730, 7 / 6)
    series = sum(c / (2 * i * (2 * i - 1)) * z ** (1 - 2 * i) for i, c in enumerate(b, 1))
    return shift + (z - 0.5) * np.log(z) - z + 0.5 * np.log(2 * np.pi) + series


def _three_j(j1, j2, j3, m1, m2, m3):
    f = math.factorial
    if not abs(j1 - j2) <= j3 <= j1 + j2 or m1 + m2 + m3 or abs(m1) > j1 or abs(m2) > j2 or abs(m3) > j3:
        return 0.0
    tri = f(j1 + j2 - j3) * f(j1 - j2 + j3) * f(-j1 + j2 + j3) / f(j1 + j2 + j3 + 1)
    pre = math.sqrt(tri * f(j1 + m1) * f(j1 - m1) * f(j2 + m2) * f(j2 - m2) * f(j3 + m3) * f(j3 - m3))
    tot = 0.0
    for k in range(j1 + j2 + j3 + 1):
        a = (k, j3 - j2 + k + m1, j3 - j1 + k - m2, j1 + j2 - j3 - k, j1 - k - m1, j2 - k + m2)
        if min(a) >= 0:
            tot += (-1) ** k / math.prod(f(i) for i in a)
    return (-1) ** (j1 - j2 - m3) * pre * tot


def _exact_template(case, seed):
    dev = _device()
    nin, nfft, qi, qf = 2048, 4096, 1.5, 0.5
    dl = math.log(10.0 / 1e-4) / (nin - 1)
    k = 1e-4 * np.exp(np.arange(nin) * dl)
    r0 = math.exp(-(nfft - 1) * dl) / 1e-4
    r = r0 * np.exp(np.arange(nfft) * dl)
    t = np.minimum(np.arange(nin), np.arange(nin)[::-1]) / (nin - 1) / 0.1
    taper = np.where(t < 1, t - np.sin(2 * np.pi * t) / (2 * np.pi), 1.0)
    x = 8 * k
    small = 1 - x * x / 10 + x ** 4 / 280
    th = np.where(x < 1e-2, small, 3 * (np.sin(x) - x * np.cos(x)) / x ** 3)
    s8w = dl * k ** 3 / (2 * np.pi ** 2) * th * th
    s8w[[0, -1]] *= 0.5

    def kernel(l, q):
        a = np.fft.fftfreq(nfft, 1.0 / nfft)
        eta = 2 * np.pi * a / (nfft * dl)
        s = q + 1j * eta
        u = np.exp((s - 2) * math.log(2) + 0.5 * math.log(math.pi) + _log_gamma(0.5 * (l + s)) -
                   _log_gamma(0.5 * (3 + l - s)) - 1j * eta * math.log(1e-4 * r0)) / nfft
        u[nfft // 2] = u[nfft // 2].real
        return torch.from_numpy(u).to(dev)

    def up(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    table, s = _window_table(seed)
    ql = np.stack([np.where(r > s[-1], 0.0, np.interp(r, s, row)) for row in table])
    edges = np.linspace(0.0, 0.2, case["bins"] + 1)
    bins = np.searchsorted(edges, k, side="right") - 1
    avg = np.stack([np.where(bins == b, k ** 3, 0.0) for b in range(case["bins"])])
    avg = avg / np.maximum(avg.sum(1, keepdims=True), 1e-300)
    avg = up((avg * 4 * np.pi * k ** -qf).T)
    th_ = _parameters(case["count"], seed)
    want = L.TEMPLATE_EB_SLOTS if case["derived"] else (1 << L.LPP_N_MOMENTS) - 1
    uinv = {l: kernel(l, qi) for l in (0, 2, 4)}
    ufwd = {l: kernel(l, qf) for l in range(0, 13, 2)}
    kd = up(k)
    out = torch.zeros((case["count"], L.LPP_N_MOMENTS, case["bins"]), device=dev, dtype=torch.float64)
    plus = ((0, 2 / 15), (2, -4 / 21), (4, 2 / 35))
    slots = ((0, 0), (1, 2), (1, 4), (1, 6), (2, 0), (2, 2), (2, 4), (3, 4), (3, 6), (3, 8), (0, 2), (0, 4), (3, 10), (3, 12))
    for c0 in range(0, case["count"], 1024):
        amp, bias, s8, tilt, gam, shot = th_[c0:c0 + 1024].T[:, :, None]
        qq = kd / gam
        tf = torch.log1p(2.34 * qq) / (2.34 * qq) * (1 + 3.89 * qq + (16.1 * qq) ** 2 + (5.46 * qq) ** 3 + (6.71 * qq) ** 4) ** -0.25
        pk = kd ** (1 + tilt) * tf * tf
        pk = pk * s8 ** 2 / (pk * up(s8w)).sum(1, keepdim=True)
        png = 1 + 12 * 100.0 * 0.17 / ((2 / 3) * kd * kd * tf * (2997.92458 ** 2 / 0.3)) if case["png"] else 1.0
        xi = {}
        for power in (0, 1, 2):
            a = torch.fft.fft(pk * png ** power * up(k ** (3 - qi) * taper), nfft)
            xi[power] = {l: (-1) ** (l // 2) * torch.fft.fft(a * uinv[l]).real * up(r ** -qi / (2 * np.pi ** 2)) for l in uinv}
            if not case["png"]:
                xi[1] = xi[2] = xi[0]
                break
        for i, (kind, l) in enumerate(slots):
            if not want >> i & 1:
                continue
            m, power = ((0, 0), (2, 1), (0, 2), (4, 2))[kind]
            terms = (((0, bias ** 2),), ((2, -amp * bias / 6),), tuple((lp, v * amp ** 2) for lp, v in plus), ((4, amp ** 2 / 420),))[kind]
            g = 0.0
            for lp, coef in terms:
                pre = (2 * l + 1) * math.sqrt(math.factorial(l - m) / math.factorial(l + m) * math.factorial(lp + m) / math.factorial(lp - m))
                win = sum(pre * _three_j(j, l, lp, 0, 0, 0) * _three_j(j, l, lp, 0, m, -m) * ql[j // 2] for j in (0, 2, 4, 6, 8))
                g = g + coef * up(win * r ** (3 - qf)) * xi[power][lp]
            f = (-1) ** (l // 2) * torch.fft.fft(torch.fft.fft(g) * ufwd[l]).real[:, :nin]
            out[c0:c0 + 1024, i] = f @ avg + (shot * 250.0 if i == 4 else 0.0) * torch.from_numpy(np.bincount(bins[(bins >= 0) & (bins < case["bins"])], minlength=case["bins"]) > 0).to(dev)
    if not case["derived"]:
        return {"native": out}

    def project(m, l, deg):
        a = np.polynomial.polynomial.polymul(_legendre_derivative(deg, m), [1, 0, -1] if m == 2 else [1, 0, -2, 0, 1])
        mu, w = np.polynomial.legendre.leggauss(20)
        v = np.polynomial.polynomial.polyval(mu, a) * np.polynomial.polynomial.polyval(mu, _legendre_derivative(l, 0))
        return float((2 * l + 1) / 2 * (w * v).sum())

    ge = [sum(project(2, l, d) * out[:, i] for i, d in ((1, 2), (2, 4), (3, 6))) for l in (0, 2)]
    mi = [sum(project(4, l, d) * out[:, i] for i, d in ((7, 4), (8, 6), (9, 8))) for l in (0, 2, 4)]
    curves = ge + [0.5 * (out[:, 4 + i] + mi[i]) for i in range(3)] + [0.5 * (out[:, 4 + i] - mi[i]) for i in range(3)]
    sigma = torch.linspace(50.0, 500.0, 8 * case["bins"], device=dev, dtype=torch.float64)
    return {"native": out, "curves": torch.cat(curves, dim=1) / sigma}


def _layers64(seed):
    return [tuple(torch.from_numpy(a).to(_device()).double() for a in layer) for layer in _network(seed)]


def _forward64(layers, x):
    for i, (w, b) in enumerate(layers):
        x = x @ w.T + b
        if i + 1 < len(layers):
            x = torch.nn.functional.gelu(x)
    return x


def _exact_predict(case, seed):
    th = _parameters(case["count"], seed)
    r = torch.tensor(RANGES, device=th.device)
    x = (2 * (th - r[:, 0]) / (r[:, 1] - r[:, 0]) - 1) * torch.tensor(FEED, device=th.device)
    mu, sd, shot, sigma, base = (torch.from_numpy(a).to(th.device) for a in _output_map(seed))
    node = -np.cos(np.pi * np.arange(NODES) / (NODES - 1))

    def basis(v):
        return torch.stack([math.prod((v - node[j]) / (node[i] - node[j]) for j in range(NODES) if j != i)
                            for i in range(NODES)], dim=1)

    l = (basis(x[:, 3])[:, :, None] * basis(x[:, 4])[:, None, :]).reshape(-1, NODES * NODES)
    u = mu + l @ base + sd * _forward64(_layers64(seed), x)
    ge, ee = th[:, :1] * th[:, 1:2], th[:, :1] ** 2
    pre = torch.cat([ge.expand(-1, 80), ee.expand(-1, 240)], dim=1) * th[:, 2:3] ** 2
    return (pre * u + th[:, 5:] * shot) / sigma


def _exact_train(case, seed):
    x, y, sched = _train_rows(case, seed)
    x, y = x.double(), y.double()
    layers = [[p.requires_grad_() for p in layer] for layer in _layers64(seed)]
    flat = [p for layer in layers for p in layer]
    mom = [[torch.zeros_like(p), torch.zeros_like(p)] for p in flat]
    losses = []
    for i in range(case["steps"]):
        rows = sched[i * case["batch"]:(i + 1) * case["batch"]].long()
        loss = ((_forward64(layers, x[rows]) - y[rows]) ** 2).mean()
        grads = torch.autograd.grad(loss, flat)
        losses.append(loss.detach())
        with torch.no_grad():
            for p, g, m in zip(flat, grads, mom):
                m[0].mul_(0.9).add_(g, alpha=0.1)
                m[1].mul_(0.999).add_(g * g, alpha=0.001)
                p -= LR * (m[0] / (1 - 0.9 ** (i + 1))) / (torch.sqrt(m[1] / (1 - 0.999 ** (i + 1))) + 1e-8)
    return {"params": np.concatenate([p.detach().reshape(-1).cpu().numpy() for p in flat]), "losses": torch.stack(losses)}


def exact(case, seed):
    k = case["kind"]
    if k == "estimate":
        pos, w, shape, ran = _estimate_inputs(case, seed)
        return _exact_estimate(case["n"], case["box"], case["tsc"], case["interlace"],
                               _edges(case["n"], case["box"], case["kfrac"], case["bins"]),
                               _observer(case["geometry"], case["box"]), case["moments"], (pos, w, shape), case["gamma"], ran)
    if k == "batch":
        out = []
        for n, pos, w, shape in _batch_inputs(case, seed):
            e = _exact_estimate(n, 1000.0, True, True, _edges(n, 1000.0, 0.8, 20), _observer("box", 1000.0), "all",
                                (pos, w, shape), False, None)
            out.append({m: e[m] for m in ("p", "raw", "norms")})
        return out
    return {"window": _exact_window, "pairs": _exact_pairs, "template": _exact_template, "predict": _exact_predict,
            "train": _exact_train}[k](case, seed)
