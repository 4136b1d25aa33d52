"""Performance cases of the LOSS library: the calls that programs built on it make, over the sizes they make them at.

Every case goes through the package's public ``Grid`` class on device-resident data:

* ``derivative``: stand-alone derivative operators along every axis of a grid;
* ``steps``: a segment of a simulation: time steps of one shot, its traces and its wavefield snapshot;
* ``survey``: a segment of a multi-shot survey: batched, graph-replayed steps of uneven shots and their traces;
* ``gradient``: seismogram misfit and model gradient of one shot from rest (one inversion iteration).

``steps`` cases carry their wavefield from one pass to the next, as a running simulation does.  Sizes are those of the
repository's standard workloads (129^2, 2049^2, 257^3, 193^3, shots of 512 to 2048 intervals) or generic ones between.
"""
import math

import numpy as np
import torch

import paper_2301_05127_gb300 as loss

H = 10.0  # grid spacing [m]


def listed():
    return [
        # one derivative of a small 2-D field: the cost of a call
        dict(name="deriv_129", kind="derivative", dim=2, nz=128, ny=0, nx=128, pz=2, py=1, px=2, n_nb=12,
             precision="fp64", second=False, adjoint=False),
        # first and second derivatives and the transpose along all axes of a 3-D field (spatial operators of a solver)
        dict(name="deriv_257cube", kind="derivative", dim=3, nz=256, ny=256, nx=256, pz=4, py=4, px=4, n_nb=20,
             precision="fp32", second=True, adjoint=True),
        # the small parity workload: a run of many short steps, FP64
        dict(name="acoustic_129_fp64", kind="steps", physics="acoustic", dim=2, nz=128, ny=0, nx=128, pz=2, py=1,
             px=2, n_nb=12, precision="fp64", steps=100, pml=20, knots=False),
        # the headline workload: layered 2049^2 model, FP32 with compensated updates
        dict(name="acoustic_2049_kahan", kind="steps", physics="acoustic", dim=2, nz=2048, ny=0, nx=2048, pz=8, py=1,
             px=8, n_nb=20, precision="fp32_kahan", steps=20, pml=40, knots=False),
        # the same step in FP64 at 1025^2 (reference-accuracy runs)
        dict(name="acoustic_1025_fp64", kind="steps", physics="acoustic", dim=2, nz=1024, ny=0, nx=1024, pz=8, py=1,
             px=8, n_nb=20, precision="fp64", steps=20, pml=40, knots=False),
        # a model whose extent is what the survey area gave: unequal sides, patch lengths that are no round number
        dict(name="acoustic_ragged_fp32", kind="steps", physics="acoustic", dim=2, nz=1098, ny=0, nx=2310, pz=9, py=1,
             px=11, n_nb=16, precision="fp32", steps=20, pml=30, knots=False),
        # a grid refined around a target: knots of their own on both axes
        dict(name="acoustic_knots_513", kind="steps", physics="acoustic", dim=2, nz=512, ny=0, nx=512, pz=8, py=1,
             px=8, n_nb=20, precision="fp32_kahan", steps=10, pml=20, knots=True),
        # a survey of uneven shots, batched, ten steps in one graph (throughput modelling)
        dict(name="survey_20", kind="survey", shots=20, lo=4, hi=16, m=128, n_nb=20, precision="fp32", steps=10,
             pml=40),
        # the 3-D elastic workload, homogeneous, FP32 with compensated updates
        dict(name="elastic_257_kahan", kind="steps", physics="elastic", dim=3, nz=256, ny=256, nx=256, pz=4, py=4,
             px=4, n_nb=20, precision="fp32_kahan", steps=4, pml=20, hetero=False, force=False),
        # the z-refined double-layer grid with a body force in FP64 (the paper's Sec. 4.3)
        dict(name="elastic_refined_fp64", kind="steps", physics="elastic", dim=3, nz=128, ny=64, nx=64, pz=4, py=2,
             px=2, n_nb=16, precision="fp64", steps=6, pml=10, hetero=True, force=True),
        # one inversion iteration of a 2-D model in FP64
        dict(name="gradient_257_fp64", kind="gradient", physics="acoustic", dim=2, nz=256, ny=0, nx=256, pz=4, py=1,
             px=4, n_nb=16, precision="fp64", steps=40, pml=20),
        # one inversion iteration of the 3-D heterogeneous elastic workload
        dict(name="gradient_193cube", kind="gradient", physics="elastic", dim=3, nz=192, ny=192, nx=192, pz=4, py=4,
             px=4, n_nb=20, precision="fp32_kahan", steps=16, pml=20),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _axis(rng, lo, hi, mlo=24, mhi=256):
    """(n, p) of one axis: n intervals between lo and hi in p patches of any length."""
    n = _log(rng, lo, hi)
    m = int(round(min(_log(rng, mlo, mhi), n)))
    p = max(1, int(round(n / m)))
    while p * m > hi:
        p -= 1
    return p * m, p


def draw(rng):
    kind = rng.choice(["derivative", "acoustic", "acoustic", "acoustic", "survey", "elastic", "elastic", "gradient2",
                       "gradient3"])
    c = {"n_nb": rng.randint(8, 22)}
    if kind in ("derivative", "acoustic", "elastic", "gradient2", "gradient3"):
        dim = {"acoustic": 2, "elastic": 3, "gradient2": 2, "gradient3": 3}.get(kind) or rng.choice([2, 3])
        lo, hi = {"acoustic": (96, 2048), "elastic": (32, 256), "gradient2": (64, 512), "gradient3": (32, 160)}.get(
            kind) or ((96, 2048) if dim == 2 else (32, 256))
        c["dim"] = dim
        c["nz"], c["pz"] = _axis(rng, lo, hi)
        c["ny"], c["py"] = _axis(rng, lo, hi) if dim == 3 else (0, 1)
        c["nx"], c["px"] = _axis(rng, lo, hi)
        c["precision"] = rng.choice(["fp64", "fp32", "fp32_kahan"])
    if kind == "derivative":
        c["precision"] = rng.choice(["fp64", "fp32"])
        c.update(kind="derivative", second=rng.random() < 0.5, adjoint=rng.random() < 0.5)
    elif kind == "acoustic":
        pts = (c["nz"] + 1) * (c["nx"] + 1)
        knots = rng.random() < 0.2
        c.update(kind="steps", physics="acoustic", steps=max(5, min(60, int(2e7 / pts))), knots=knots,
                 pml=min(rng.randint(10, 40), c["nz"] // 3, c["nx"] // 3))
        if knots:  # pulses that the refined grid resolves
            c["steps"] = min(c["steps"], 10)
    elif kind == "survey":
        lo = rng.randint(4, 8)
        c.update(kind="survey", shots=rng.randint(3, 20), lo=lo, hi=lo + rng.randint(2, 8), m=rng.choice([64, 96, 128]),
                 precision=rng.choice(["fp32", "fp32_kahan"]), steps=rng.randint(4, 10), pml=rng.randint(20, 40))
    elif kind == "elastic":
        pts = (c["nz"] + 1) * (c["ny"] + 1) * (c["nx"] + 1)
        c.update(kind="steps", physics="elastic", steps=max(2, min(12, int(4e7 / pts))),
                 pml=min(rng.randint(6, 20), c["nz"] // 3, c["ny"] // 3, c["nx"] // 3), hetero=rng.random() < 0.6,
                 force=rng.random() < 0.3)
    else:
        el = kind == "gradient3"
        c.update(kind="gradient", physics="elastic" if el else "acoustic", steps=rng.randint(8, 16) if el else
                 rng.randint(16, 60), pml=min(rng.randint(6, 20), c["nz"] // 3, c["nx"] // 3, *([c["ny"] // 3] if el else [])))
    c["n_nb"] = min([c["n_nb"]] + [c[n] // c[p] for n, p in (("nz", "pz"), ("ny", "py"), ("nx", "px")) if c.get(n)])
    return c


# ----------------------------------------------------------------------------------------------------------------
# Inputs.
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _shape(c):
    return (c["nz"] + 1, c["nx"] + 1) if c["dim"] == 2 else (c["nz"] + 1, c["ny"] + 1, c["nx"] + 1)


def _axes(c):
    return [("nz", "pz"), ("nx", "px")] if c["dim"] == 2 else [("nz", "pz"), ("ny", "py"), ("nx", "px")]


def _outer(vs):
    out = vs[0]
    for v in vs[1:]:
        out = out[..., None] * v
    return out


def _pulses(rng, shape, amp, count=5, near=None):
    """A smooth wavefield: Gaussian pulses of 4 to 8 cells at random places, of either sign; the first of them passes
    the plane ``near`` of axis 0 (the receivers' plane)."""
    f = torch.zeros(shape, dtype=torch.float64, device=_dev())
    for k in range(count):
        w = rng.uniform(4.0, 8.0)
        vs = []
        for a, n in enumerate(shape):
            c = rng.uniform(0.2, 0.8) * (n - 1)
            if k == 0 and a == 0 and near is not None:
                c = near + rng.uniform(0.0, 8.0)
            x = torch.arange(n, dtype=torch.float64, device=_dev()) - c
            vs.append(torch.exp(-x * x / (2.0 * w * w)))
        f += amp * rng.uniform(-1.0, 1.0) * _outer(vs)
    return f


def _smooth(rng, shape, count=6):
    """A smooth random perturbation in about -1 .. 1 (products of cosines with wavelengths from 20 cells up)."""
    f = torch.zeros(shape, dtype=torch.float64, device=_dev())
    for _ in range(count):
        vs = [torch.cos(torch.arange(n, dtype=torch.float64, device=_dev()) * rng.uniform(0.05, 0.3) +
                        rng.uniform(0.0, 6.28)) for n in shape]
        f += _outer(vs) / math.sqrt(count)
    return f.clamp(-2.0, 2.0)


def _layers(shape, speeds, bounds):
    z = torch.arange(shape[0], device=_dev(), dtype=torch.float64) / (shape[0] - 1)
    v = torch.tensor(speeds, dtype=torch.float64, device=_dev())
    v = v[torch.searchsorted(torch.tensor(bounds, dtype=torch.float64, device=_dev()), z, right=True)]
    return v.reshape([-1] + [1] * (len(shape) - 1)).expand(shape)


def _model(c, rng):
    """(vp, vs, rho): layered with a 5 % perturbation in 2-D, constant or perturbed in 3-D."""
    shape = _shape(c)
    one = torch.ones(shape, dtype=torch.float64, device=_dev())
    if c["physics"] == "acoustic":
        vp = _layers(shape, [1500.0, 2500.0, 3500.0], [1 / 3, 2 / 3]) * (1.0 + 0.05 * _smooth(rng, shape))
        rho = 1000.0 * (1.0 + 0.05 * _smooth(rng, shape)) if c["kind"] == "gradient" else 1000.0 * one
        return vp.contiguous(), None, rho.contiguous()
    if not c.get("hetero", True):
        return 3000.0 * one, 1730.0 * one, 2000.0 * one
    return tuple((m * (1.0 + 0.05 * _smooth(rng, shape))).contiguous() for m in (3000.0, 1730.0, 2000.0))


def _knots(n):
    """Knots on [0, 10 n]: spacings from 0.7 to 1.3 times 10 m, finest in the middle."""
    s = np.arange(n + 1) / n
    return H * n * (s + 0.3 * np.sin(2.0 * np.pi * s) / (2.0 * np.pi))


def _setup(c, seed):
    """Everything that a program knows of one shot: model, source, receivers, wavefield, layer, time step."""
    rng = np.random.default_rng(seed)
    shape = _shape(c)
    el = c["physics"] == "elastic"
    vp, vs, rho = _model(c, rng)
    vmax = float(vp.max())
    dt = 0.4 * H / vmax * (0.7 if c.get("knots") else 1.0)
    pml = c["pml"]
    grad = c["kind"] == "gradient"
    u = {"vp": vp, "vs": vs, "rho": rho, "vmax": vmax, "dt": dt, "f0": 20.0, "shape": shape, "el": el}
    plane = int(np.prod(shape[1:]))
    top = pml * plane + np.arange(plane, dtype=np.int64)
    u["receivers"] = {"sigma": top} if not el else ({"v3": top} if grad else {"v1": top, "v2": top, "v3": top})
    # source: at the centre, or (gradient, so that the few steps reach the receivers) just below the receivers
    u["src"] = tuple(s // 2 for s in shape) if not grad else (min(pml + 5, shape[0] - 1),) + tuple(s // 2 for s in shape[1:])
    u["kinds"] = () if c.get("knots") else (("pressure",) if not el else (
        ("force_x", "force_y", "force_z") if c.get("force") else ("explosive", "shear_xz")))
    u["t0"] = (c["steps"] * 0.4 * dt) if grad else 1.2 / u["f0"]
    rate = 50.0 * (1.0 if not c.get("force") else 1.0 / H)  # stress rate (or force) at the centre, times t
    u["amp"] = rate * H ** len(shape) * (2.0 * math.pi * 4.0) ** (len(shape) / 2)
    fields = (("sigma", "v1", "v3") if not el else
              ("v1", "v2", "v3", "s11", "s22", "s33", "s12", "s13", "s23"))
    z = 2000.0 * 2000.0  # impedance scale: stress over velocity
    dtype = torch.float64 if c["precision"] == "fp64" else torch.float32
    u["fields"] = {} if grad else {f: _pulses(rng, shape, 1.0 / z if f[0] == "v" else 1.0, near=pml).to(dtype)
                                  for f in fields}
    if grad:
        n_r = sum(len(r) for r in u["receivers"].values())
        scale = 0.2 * rate * dt * c["steps"] / (z if el else 1.0)
        t = np.arange(c["steps"])[:, None] * dt
        off = np.cos(rng.uniform(0.02, 0.2) * np.arange(n_r)[None, :] + 300.0 * t + rng.uniform(0, 6.28))
        u["d_obs"] = torch.from_numpy(scale * off).to(_dev())
    return u


def _grid(c, u):
    el = u["el"]
    n = [c[a] for a, _ in _axes(c)]
    p = [c[b] for _, b in _axes(c)]
    desc = loss.make_desc(c["dim"], loss.LOSS_ELASTIC if el else loss.LOSS_ACOUSTIC, loss.PRECISIONS[c["precision"]],
                          c["n_nb"], n, p, [H] * c["dim"], u["dt"])
    g = loss.Grid([desc])
    if c.get("knots"):
        for axis in range(c["dim"]):
            g.set_coordinates(0, axis, _knots(n[axis]))
    g.set_model(0, u["vp"], u["vs"], u["rho"])
    if u["kinds"]:
        mask = sum(loss.SOURCE_KINDS[k] for k in u["kinds"])
        idx = u["src"] if c["dim"] == 3 else (u["src"][0], 0, u["src"][1])
        g.set_source(0, idx, mask, u["amp"], u["f0"], u["t0"])
    for f, idx in u["receivers"].items():
        g.set_receivers(0, f, idx)
    g.set_pml(0, c["pml"], 1e-6, 1.0, u["f0"])
    for f, a in u["fields"].items():
        g.set_field(0, f, a)
    return g


def _shots(c, seed):
    """The shots of a survey: uneven square grids of lo .. hi patches of m intervals, 3 to 5 layers."""
    rng = np.random.default_rng(seed)
    # the first two shots take the ends of the range, the others any size between
    counts = [c["hi"], c["lo"]] + [int(k) for k in np.random.default_rng(7).integers(c["lo"], c["hi"] + 1, c["shots"])]
    out = []
    for k in counts[:c["shots"]]:
        n = k * c["m"]
        layers = int(rng.integers(3, 6))
        v = np.sort(rng.uniform(1500.0, 4000.0, layers))
        b = np.sort(rng.uniform(0.1, 0.9, layers - 1))
        out.append(dict(n=n, p=k, speeds=[float(x) for x in v], bounds=[float(x) for x in b], vmax=float(v.max()),
                        dt=0.4 * H / float(v.max()), shape=(n + 1, n + 1), f0=20.0, t0=1.2 / 20.0,
                        amp=50.0 * H * H * 2.0 * math.pi * 4.0, src=(c["pml"] + 5, n // 2), seed=int(rng.integers(1 << 30))))
    return out


def _shot_inputs(c, s):
    rng = np.random.default_rng(s["seed"])
    f = {k: _pulses(rng, s["shape"], 1.0 if k == "sigma" else 1.0 / 4e6, 3, near=c["pml"]).to(torch.float32)
         for k in ("sigma", "v1", "v3")}
    row = c["pml"] * s["shape"][1] + np.arange(s["shape"][1], dtype=np.int64)
    return _layers(s["shape"], s["speeds"], s["bounds"]).contiguous(), f, row


def prepare(case, seed):
    c = case
    if c["kind"] == "derivative":
        n = [c[a] for a, _ in _axes(c)]
        desc = loss.make_desc(c["dim"], loss.LOSS_ACOUSTIC, loss.PRECISIONS[c["precision"]], c["n_nb"], n,
                              [c[b] for _, b in _axes(c)], [H] * c["dim"], 1e-3)
        return {"case": c, "grid": loss.Grid([desc]), "f": _deriv_field(c, seed)}
    if c["kind"] == "survey":
        shots = _shots(c, seed)
        g = loss.Grid([loss.make_desc(2, loss.LOSS_ACOUSTIC, loss.PRECISIONS[c["precision"]], c["n_nb"], (s["n"], s["n"]),
                                      (s["p"], s["p"]), (H, H), s["dt"]) for s in shots])
        for k, s in enumerate(shots):
            vp, f, row = _shot_inputs(c, s)
            g.set_model(k, vp, None, torch.full_like(vp, 1000.0))
            g.set_source(k, (s["src"][0], 0, s["src"][1]), loss.LOSS_SRC_PRESSURE, s["amp"], s["f0"], s["t0"])
            g.set_receivers(k, "sigma", row)
            g.set_pml(k, c["pml"], 1e-6, 1.0, s["f0"])
            for name, a in f.items():
                g.set_field(k, name, a)
        g.set_schedule(True, c["steps"])
        return {"case": c, "grid": g, "sigma": [torch.empty(s["shape"], dtype=torch.float32, device="cuda") for s in shots]}
    u = _setup(c, seed)
    g = _grid(c, u)
    if c["kind"] == "gradient":
        return {"case": c, "grid": g, "d_obs": u["d_obs"]}
    return {"case": c, "grid": g, "out": {f: torch.empty_like(a) for f, a in u["fields"].items()}}


def _deriv_field(c, seed):
    rng = np.random.default_rng(seed)
    dtype = torch.float64 if c["precision"] == "fp64" else torch.float32
    return (_smooth(rng, _shape(c)) + _pulses(rng, _shape(c), 1.0)).to(dtype)


def run(state):
    c, g = state["case"], state["grid"]
    if c["kind"] == "derivative":
        out = {}
        for axis in range(c["dim"]):
            out["d%d" % axis] = g.derivative(0, axis, state["f"], second=c["second"])
            if c["adjoint"]:
                out["t%d" % axis] = g.derivative_adjoint(0, axis, state["f"])
        return out
    if c["kind"] == "gradient":
        misfit, grads = g.gradient(0, state["d_obs"], c["steps"])
        return {"misfit": misfit, "vp": grads["vp"], "vs": grads["vs"], "rho": grads["rho"]}
    g.step(c["steps"])
    if c["kind"] == "survey":
        traces = [g.record(k)["_all"] for k in range(c["shots"])]
        for k in range(c["shots"]):
            g.get_field(k, "sigma", out=state["sigma"][k])
        return {"traces": traces, "sigma": state["sigma"]}
    out = {f: g.get_field(0, f, out=a) for f, a in state["out"].items()}
    out["traces"] = g.record(0)["_all"]
    return out


# ----------------------------------------------------------------------------------------------------------------
# What a pass cannot do without.
def work(case):
    c = case
    es = 8 if c["precision"] == "fp64" else 4
    comp = c["precision"] == "fp32_kahan"
    taps = 2 * (2 * c["n_nb"] + 1)

    def line(n, p):  # flops of one derivative per point: two recurrences and the junction sums
        return 8.0 + taps * (p + 1) / (n + 1)

    if c["kind"] == "survey":
        k = (c["lo"] + c["hi"]) / 2.0
        pts = float(c["shots"]) * (k * c["m"] + 1) ** 2
        return {"bytes": pts * c["steps"] * es * (7 + (6 if comp else 0)), "flops": pts * c["steps"] * (4 * line(k * c["m"], k) + 12)}
    pts = float(np.prod(_shape(c)))
    dflops = sum(line(c[a], c[b]) for a, b in _axes(c))
    if c["kind"] == "derivative":
        outs = c["dim"] * (1 + int(c["second"]) + int(c["adjoint"]))
        return {"bytes": pts * es * (1 + outs), "flops": pts * dflops * (outs / c["dim"])}
    el = c["physics"] == "elastic"
    nf = 9 if el else 3
    model = (3 if c.get("hetero", True) else 0) if el else (2 if c["kind"] == "gradient" else 1)
    step_b = es * (2 * nf * (2 if comp else 1) + model)
    step_f = dflops * (6 if el else 2) + (60 if el else 12)
    if c["kind"] == "gradient":  # forward run, then per step the forward state again and the adjoint state
        return {"bytes": pts * c["steps"] * (step_b + es * (3 * nf + model)) + pts * 8 * (4 + 2 * int(el)),
                "flops": pts * c["steps"] * 3 * step_f}
    return {"bytes": pts * c["steps"] * step_b, "flops": pts * c["steps"] * step_f}


# ----------------------------------------------------------------------------------------------------------------
# The same results in 64 bits: the derivative as a dense matrix per axis, the time step as the paper writes it.
def _spline_matrix(n, p, n_nb, h, second=False):
    """(n + 1)^2 matrices of the first (and second) LOSS derivative along a line of n intervals in p patches."""
    f8 = dict(dtype=torch.float64, device=_dev())
    m = n // p

    def band(size, end):
        a = torch.zeros(size + 3, size + 3, **f8)
        i = torch.arange(size + 1, device=_dev())
        a[i + 1, i], a[i + 1, i + 1], a[i + 1, i + 2] = 1 / 6, 4 / 6, 1 / 6
        a[0, :3] = torch.tensor(end, **f8)
        a[-1, -3:] = torch.tensor(end, **f8)
        return a

    inv = torch.linalg.inv(band(n, [1 / h**2, -2 / h**2, 1 / h**2]))[:, 1:n + 2]  # coefficients from samples
    w = torch.zeros(p + 1, n + 1, **f8)
    for j in range(p + 1):
        q = j * m
        lo = q if j == 0 else max(0, q - n_nb)
        hi = q if j == p else min(n, q + n_nb)
        w[j, lo:hi + 1] = ((inv[q + 2] - inv[q]) / (2.0 * h))[lo:hi + 1]
    loc = torch.linalg.inv(band(m, [-1 / (2 * h), 0.0, 1 / (2 * h)]))
    ops = [(loc[2:] - loc[:-2]) / (2 * h)] + ([(loc[:-2] - 2 * loc[1:-1] + loc[2:]) / h**2] if second else [])
    out = []
    for e in ops:
        d = torch.zeros(n + 1, n + 1, **f8)
        cnt = torch.zeros(n + 1, 1, **f8)
        for k in range(p):
            rows = slice(k * m, k * m + m + 1)
            d[rows] += e[:, :1] * w[k] + e[:, -1:] * w[k + 1]
            d[rows, rows] += e[:, 1:-1]
            cnt[rows] += 1.0
        out.append(d / cnt)
    return out if second else out[0]


def _knot_matrix(x, p, n_nb):
    """(n + 1)^2 matrix of the LOSS derivative on the knots x: slopes of the patched cubic spline."""
    n = len(x) - 1
    m = n // p
    h = np.diff(x)
    t, r = np.zeros((n + 1, n + 1)), np.zeros((n + 1, n + 1))
    t[0, :2], r[0, :2] = (2.0, 1.0), (-3.0 / h[0], 3.0 / h[0])
    t[n, n - 1:], r[n, n - 1:] = (1.0, 2.0), (-3.0 / h[-1], 3.0 / h[-1])
    for i in range(1, n):
        a, b = 3.0 * h[i] / h[i - 1], 3.0 * h[i - 1] / h[i]
        t[i, i - 1:i + 2] = (h[i], 2.0 * (h[i - 1] + h[i]), h[i - 1])
        r[i, i - 1:i + 2] = (-a, a - b, b)
    t, r = (torch.from_numpy(v).to(_dev()) for v in (t, r))
    full = torch.linalg.solve(t, r)
    d = torch.zeros_like(full)
    for j in range(p + 1):
        q = j * m
        lo = q if j == 0 else max(0, q - n_nb)
        hi = q if j == p else min(n, q + n_nb)
        d[q, lo:hi + 1] = full[q, lo:hi + 1]
    for k in range(p):
        i = slice(k * m + 1, (k + 1) * m)
        rhs = r[i] - t[i, k * m:k * m + 1] * d[k * m] - t[i, (k + 1) * m:(k + 1) * m + 1] * d[(k + 1) * m]
        d[i] = torch.linalg.solve(t[i, i], rhs)
    return d


def _along(d, f, axis):
    if axis == f.dim() - 1:
        return f @ d.T
    if axis == 0:
        return (d @ f.reshape(f.shape[0], -1)).reshape(f.shape)
    return torch.matmul(d, f)


class _Layer:
    """Coefficients of the absorbing layer's exact sub-flow over tau along one axis, broadcastable."""

    def __init__(self, n, width, tau, vmax, f0, axis, dim, x=None):
        x = H * np.arange(n + 1) if x is None else x
        r, d = np.zeros(n + 1), np.zeros(n + 1)
        for inner, end, sl in ((x[width], x[0], slice(0, width)), (x[n - width], x[n], slice(n - width + 1, n + 1))):
            depth = abs(end - inner)
            r[sl] = np.abs(x[sl] - inner) / depth
            d[sl] = -3.0 * vmax * math.log(1e-6) / (2.0 * depth) * r[sl] ** 2
        alpha = math.pi * f0 * (1.0 - r)
        beta = np.where(d > 0, d + alpha, 1.0)
        e = np.exp(-beta * tau)
        cols = (np.where(d > 0, e, 0.0), np.where(d > 0, d * (1.0 - e) / beta, 0.0), np.where(d > 0, 1.0 / beta, 0.0),
                np.where(d > 0, tau * alpha / (d + alpha + (d == 0)), tau))
        shape = [1] * dim
        shape[axis] = -1
        self.e, self.q, self.ib, self.c = (torch.from_numpy(v).reshape(shape).to(_dev()) for v in cols)

    def __call__(self, mem, g):
        """(new memory variable, increment factor) for the frozen derivative g."""
        new = self.e * mem - self.q * g
        return new, self.ib * (new - mem) - self.c * g


def _simulate(c, u, model=None):
    """Literal Strang steps; returns (fields, traces [steps][receivers])."""
    dim, el, dt, shape = c["dim"], u["el"], u["dt"], u["shape"]
    vp, vs, rho = (u["vp"], u["vs"], u["rho"]) if model is None else model
    axes = _axes(c)
    xs = [_knots(c[a]) if c.get("knots") else None for a, _ in axes]
    ds = [_knot_matrix(x, c[b], c["n_nb"]) if x is not None else _spline_matrix(c[a], c[b], c["n_nb"], H)
          for (a, b), x in zip(axes, xs)]
    lay = {tau: [_Layer(c[a], c["pml"], tau, u["vmax"], u["f0"], k, dim, xs[k]) for k, (a, _) in enumerate(axes)]
           for tau in (0.5 * dt, dt)}
    comps = {1: dim - 1, 2: 1, 3: 0}  # component -> array axis
    names = [1, 2, 3] if dim == 3 else [1, 3]
    zero = torch.zeros(shape, dtype=torch.float64, device=_dev())
    allf = ("v1", "v2", "v3", "s11", "s22", "s33", "s12", "s13", "s23") if el else ("sigma", "v1", "v3")
    st = {f: u["fields"][f].double() if f in u["fields"] else zero for f in allf}
    mem = {}
    b = 1.0 / rho
    lam, mu = (rho * (vp * vp - 2.0 * vs * vs), rho * vs * vs) if el else (rho * vp * vp, None)
    prof = None
    if u["kinds"]:
        gs = [torch.exp(-(torch.arange(n, dtype=torch.float64, device=_dev()) - s) ** 2 / 8.0) *
              ((torch.arange(n, device=_dev()) - s).abs() <= 12) for n, s in zip(shape, u["src"])]
        prof = _outer(gs)
        prof = prof * (u["amp"] / (float(prof.sum()) * H ** dim))

    def ricker(t):
        a = (math.pi * u["f0"] * (t - u["t0"])) ** 2
        return (1.0 - 2.0 * a) * math.exp(-a)

    def flow(key, f, comp, tau):
        k = comps[comp]
        mem[key], x = lay[tau][k](mem.get(key, zero), _along(ds[k], f, k))
        return x

    def half_a(tau, t):
        for i in names:
            if el:
                s = {j: st["s%d%d" % (min(i, j), max(i, j))] for j in names}
                acc = -sum(flow("psi%d%d" % (i, j), s[j], j, tau) for j in names)
                if "force_" + " xyz"[i] in u["kinds"]:
                    acc = acc + tau * ricker(t) * prof
            else:
                acc = flow("psi%d" % i, st["sigma"], i, tau)
            st["v%d" % i] = st["v%d" % i] + b * acc

    def full_b(t):
        if not el:
            st["sigma"] = st["sigma"] + lam * sum(flow("phi%d" % i, st["v%d" % i], i, dt) for i in names)
            if "pressure" in u["kinds"]:
                st["sigma"] = st["sigma"] + dt * ricker(t) * prof
            return
        x = {(i, j): -flow("phi%d%d" % (i, j), st["v%d" % i], j, dt) for i in names for j in names}
        tr = x[1, 1] + x[2, 2] + x[3, 3]
        s = dt * ricker(t) * prof if prof is not None else None
        for i in names:
            k = "s%d%d" % (i, i)
            st[k] = st[k] + (lam * tr + 2.0 * mu * x[i, i]) + (s if "explosive" in u["kinds"] else 0.0)
        for i, j in ((1, 2), (1, 3), (2, 3)):
            k = "s%d%d" % (i, j)
            st[k] = st[k] + mu * (x[i, j] + x[j, i]) + (s if k == "s13" and "shear_xz" in u["kinds"] else 0.0)

    order = ["v1", "v2", "v3", "sigma"]
    rec = [(f, torch.from_numpy(u["receivers"][f]).to(_dev())) for f in order if f in u["receivers"]]
    traces = []
    for n in range(c["steps"]):
        half_a(0.5 * dt, n * dt)
        full_b((n + 0.5) * dt)
        half_a(0.5 * dt, (n + 1) * dt)
        traces.append(torch.cat([st[f].reshape(-1)[i] for f, i in rec]))
    return st, torch.stack(traces)


def exact(case, seed):
    c = case
    if c["kind"] == "derivative":
        f = _deriv_field(c, seed).double()
        out = {}
        for axis, (a, b) in enumerate(_axes(c)):
            d1, d2 = _spline_matrix(c[a], c[b], c["n_nb"], H, second=True)
            out["d%d" % axis] = (_along(d1, f, axis), _along(d2, f, axis)) if c["second"] else _along(d1, f, axis)
            if c["adjoint"]:
                out["t%d" % axis] = _along(d1.T, f, axis)
        return out
    if c["kind"] == "survey":
        sig, tr = [], []
        for s in _shots(c, seed):
            vp, f, row = _shot_inputs(c, s)
            cc = dict(dim=2, nz=s["n"], nx=s["n"], pz=s["p"], px=s["p"], n_nb=c["n_nb"], pml=c["pml"], steps=c["steps"])
            u = dict(s, vp=vp, vs=None, rho=torch.full_like(vp, 1000.0), fields=f, receivers={"sigma": row},
                     kinds=("pressure",), el=False)
            st, t = _simulate(cc, u)
            sig.append(st["sigma"])
            tr.append(t)
        return {"traces": tr, "sigma": sig}
    u = _setup(c, seed)
    if c["kind"] == "gradient":
        m = [None if v is None else v.clone().requires_grad_() for v in (u["vp"], u["vs"], u["rho"])]
        _, tr = _simulate(c, u, m)
        j = 0.5 * ((tr - u["d_obs"]) ** 2).sum()
        j.backward()
        return {"misfit": float(j.detach()), "vp": m[0].grad, "vs": None if m[1] is None else m[1].grad, "rho": m[2].grad}
    st, tr = _simulate(c, u)
    return {**{f: st[f] for f in u["fields"]}, "traces": tr}
