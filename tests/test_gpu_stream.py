"""GPU parity of the barrier-free engines (column and row kernels) at the edges of their geometry: rows of one and
several windows, a last chunk of 1, 9 and other lengths, lines of one and several segments, patches at the shortest
length they take, layers and receivers inside them.  Oracle: the FP64 Strang step.  Tolerances are those of the
other run tests: 1e-12 (FP64), 1e-5 (FP32)."""
import dataclasses
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from oracle.wave import ELASTIC_FIELDS, Simulation  # noqa: E402
from synth import acoustic2d_small, elastic3d_homogeneous  # noqa: E402
from synth.workloads import random_field  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp32_kahan": 1e-5}


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as ge

    ge.build()
    import paper_2301_05127_gb300 as p

    return p


# (n, p, n_nb) per axis z, y, x: one 9-point last chunk and one-patch axes; two and more row windows; a row of 1 + 8 k
# points more than a window; patches of 24 and 30 points; rows of 8- and 16-lane groups
ELASTIC = [((40, 40, 40), (1, 1, 1), 8), ((48, 41, 262), (2, 1, 2), 20), ((60, 40, 256), (2, 1, 8), 16),
           ((90, 44, 65), (3, 1, 1), 13), ((42, 130, 120), (1, 5, 4), 22)]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_kahan"])
@pytest.mark.parametrize("geom", range(len(ELASTIC)))
def test_elastic_step(pkg, prec, geom):
    n, p, n_nb = ELASTIC[geom]
    shape = tuple(k + 1 for k in n)
    w = elastic3d_homogeneous(n=32, p=2, n_nb=n_nb, steps=6, pml_width=7, precision=prec)
    hetero = geom % 2 == 1

    def model():
        if not hetero:
            return np.full(shape, 3000.0), np.full(shape, 1730.0), np.full(shape, 2000.0)
        return tuple(v * (1.0 + 0.05 * random_field(shape, s, 3.0)) for v, s in ((3000.0, 1), (1730.0, 2), (2000.0, 3)))

    vp = model()[0].max()
    kinds = ("explosive", "shear_xz") if geom % 3 else ("force_x", "force_y", "force_z", "explosive")
    rec = np.concatenate([np.arange(shape[2]) + 3 * shape[1] * shape[2], np.arange(0, int(np.prod(shape)), 997)])
    w = dataclasses.replace(w, n=n, p=p, model_fn=model, src_index=tuple(k // 2 for k in n), src_kinds=kinds, f0=40.0,
                            t0=0.002, dt=0.4 * 10.0 / vp, receivers={"v1": rec, "v3": rec, "s13": rec})
    rng = np.random.default_rng(5)
    g = pkg.Grid.from_workloads([w], precision=prec)
    sim = Simulation(w)
    for f in ELASTIC_FIELDS:  # a smooth wavefield that fills the grid
        a = random_field(shape, int(rng.integers(1 << 30)), 3.0) * (1e-7 if f[0] == "v" else 1.0)
        a = a.astype(np.float32 if prec != "fp64" else np.float64)
        g.set_field(0, f, a)
        sim.state[f] = a.astype(np.float64)
    g.step(w.steps)
    sim.step(w.steps)
    for f in ELASTIC_FIELDS:
        ref = sim.state[f]
        err = np.linalg.norm(g.get_field(0, f).astype(np.float64) - ref) / np.linalg.norm(ref)
        assert err < TOL[prec], (f, err)
    tr = g.record(0)
    for f in w.receivers:
        ref = sim.trace_array(f)
        scale = np.abs(sim.state[f]).max()
        assert np.abs(tr[f] - ref).max() / scale < 10 * TOL[prec], f
    g.close()


# rows of 8-, 16- and 32-lane groups, of one window with and without a ninth point, of two and three windows; short last
# chunks; lines of several segments; FP32 rows that the pipelined kernel does not take (patches of 2 k + 1 points)
ACOUSTIC = [((40, 44), (1, 1), 8), ((96, 128), (2, 4), 12), ((57, 256), (1, 8), 20), ((130, 264), (2, 4), 16),
            ((64, 600), (1, 5), 20), ((700, 71), (4, 1), 9), ((44, 513), (1, 9), 16)]


def _acoustic(pkg, n, p, n_nb, prec, seed, steps=8, pml=9):
    shape = tuple(k + 1 for k in n)
    vp = 2000.0 * (1.0 + 0.05 * random_field(shape, seed, 4.0))
    rho = 1000.0 * (1.0 + 0.05 * random_field(shape, seed + 1, 4.0)) if seed % 2 else np.full(shape, 1000.0)
    rec = np.concatenate([np.arange(shape[1]) + 3 * shape[1], np.arange(0, int(np.prod(shape)), 97)])
    w = acoustic2d_small(n=32, p=1, n_nb=n_nb, steps=steps, pml_width=pml)
    return dataclasses.replace(w, n=n, p=p, precision=prec, dt=0.4 * 10.0 / vp.max(), model_fn=lambda: (vp, None, rho),
                               src_index=(n[0] // 2, n[1] - 2), f0=40.0, t0=0.002, amp=1e4,
                               receivers={"sigma": rec, "v1": rec, "v3": rec})


def _fields(w, prec, seed):
    dt = np.float64 if prec == "fp64" else np.float32
    return {f: (random_field(w.shape, seed + k, 4.0) * (1.0 if f == "sigma" else 5e-7)).astype(dt)
            for k, f in enumerate(("sigma", "v1", "v3"))}


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_kahan"])
@pytest.mark.parametrize("geom", range(len(ACOUSTIC)))
def test_acoustic_step(pkg, prec, geom):
    n, p, n_nb = ACOUSTIC[geom]
    w = _acoustic(pkg, n, p, n_nb, prec, 10 + geom)
    init = _fields(w, prec, 50 + geom)
    g = pkg.Grid.from_workloads([w], precision=prec)
    sim = Simulation(w)
    for f, a in init.items():
        g.set_field(0, f, a)
        sim.state[f] = a.astype(np.float64)
    g.step(w.steps)
    sim.step(w.steps)
    for f in init:
        ref = sim.state[f]
        err = np.linalg.norm(g.get_field(0, f).astype(np.float64) - ref) / np.linalg.norm(ref)
        assert err < TOL[prec], (f, err)
    tr = g.record(0)
    for f in w.receivers:
        ref = sim.trace_array(f)
        assert np.abs(tr[f] - ref).max() / np.abs(ref).max() < 10 * TOL[prec], f
    g.close()


@pytest.mark.parametrize("graph", [0, 3])
@pytest.mark.parametrize("mixed", [False, True])
def test_batched_fp64_equals_per_shot(pkg, graph, mixed):
    """All FP64 shots of a handle in one launch per kernel: the per-shot schedule's fields and traces bit for bit, also
    with a shot whose patches are too short for the engines (the handle then goes per shot)."""
    geoms = [ACOUSTIC[1], ACOUSTIC[3], ACOUSTIC[0], ACOUSTIC[4]] + ([((36, 36), (3, 3), 6)] if mixed else [])
    ws = [_acoustic(pkg, n, p, n_nb, "fp64", 30 + k) for k, (n, p, n_nb) in enumerate(geoms)]
    res = []
    for batched in (True, False):
        g = pkg.Grid.from_workloads(ws)
        g.set_schedule(batched, graph if batched else 0)
        for s, w in enumerate(ws):
            for f, a in _fields(w, "fp64", 70 + s).items():
                g.set_field(s, f, a)
        g.step(3)
        g.get_field(0, "v1")  # back to the integer time level in between
        g.step(7)
        res.append([[g.get_field(s, f) for f in ("sigma", "v1", "v3")] + [g.record(s)["_all"]] for s in range(len(ws))])
        g.close()
    for s in range(len(ws)):
        for a, b in zip(res[0][s], res[1][s]):
            assert np.array_equal(a, b), s


# (n, p, n_nb) of two or three axes: segments of 40 positions and more, two row windows, a 9-point last chunk, the
# shortest line and patch, patches that overlap in three junctions' reach, odd row lengths (unaligned rows)
OPERATORS = [((40, 41), (1, 1), 8), ((257, 510), (1, 17), 20), ((512, 264), (16, 8), 12), ((44, 40, 63), (1, 2, 1), 9),
             ((120, 48, 72), (5, 2, 3), 16)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("geom", range(len(OPERATORS)))
def test_derivative_operators(pkg, prec, geom):
    """First and second derivative and the transpose against the oracle (tolerances of the derivative tests), device
    arrays at an odd element offset; written over their input they give the same."""
    import torch

    from oracle import spline

    n, p, n_nb = OPERATORS[geom]
    h = tuple(1.0 + 0.5 * k for k in range(len(n)))
    t1, t2 = (1e-12, 1e-11) if prec == "fp64" else (2e-5, 2e-4)
    g = pkg.Grid([pkg.make_desc(len(n), pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[prec], n_nb, n, p, h, 1e-3)])
    rng = np.random.default_rng(geom)
    f = (rng.standard_normal(g.shape()) + 5.0 * np.sin(np.linspace(0, 9, g.shape()[-1]))).astype(g.dtype)
    dev = torch.empty(f.size + 1, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")[1:]
    dev = dev.view(f.shape)
    dev.copy_(torch.from_numpy(f))
    for axis in range(len(n)):
        r1, r2 = spline.derivative(f.astype(np.float64), axis, n[axis], p[axis], h[axis], n_nb, second=True)
        d1, d2 = (v.cpu().numpy() for v in g.derivative(0, axis, dev, second=True))
        only = g.derivative(0, axis, dev).cpu().numpy()
        assert np.abs(d1 - r1).max() < t1 * np.abs(r1).max(), axis
        assert np.abs(only - r1).max() < t1 * np.abs(r1).max(), axis
        assert np.abs(d2 - r2).max() < t2 * np.abs(r2).max(), axis
        eye = np.eye(n[axis] + 1)
        D = spline.derivative(eye, 0, n[axis], p[axis], h[axis], n_nb)
        D = D[0] if isinstance(D, tuple) else D
        rt = np.moveaxis(np.tensordot(D.T, f.astype(np.float64), axes=(1, axis)), 0, axis)
        t = g.derivative_adjoint(0, axis, dev).cpu().numpy()
        assert np.abs(t - rt).max() < t1 * np.abs(rt).max(), axis
        over = dev.clone()
        assert pkg.lib().loss_derivative(g.h, 0, axis, over.data_ptr(), over.data_ptr(), None, pkg.LOSS_MEM_DEVICE) == 0
        g.sync()
        assert np.abs(over.cpu().numpy() - r1).max() < t1 * np.abs(r1).max(), axis
    g.close()


@pytest.mark.parametrize("graph", [0, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp32_kahan"])
def test_batched_long_rows(pkg, prec, graph):
    """FP32 rows of 513 points and more in one launch for all shots (row engine): the per-shot schedule's bits, and the
    fields of the pipelined row kernel (the items family's rounding apart) to the run tolerance."""
    geoms = [((64, 512), (2, 4), 20), ((96, 1024), (3, 8), 12), ((48, 520), (1, 13), 16)]
    ws = [_acoustic(pkg, n, p, n_nb, prec, 50 + k) for k, (n, p, n_nb) in enumerate(geoms)]
    res = []
    for mode in range(3):
        g = pkg.Grid.from_workloads(ws)
        g.set_schedule(mode == 0, graph if mode == 0 else 0)
        if mode == 2:
            g.set_wait_limit(1 << 20)  # a limit of one's own keeps the kernel that waits
        for s, w in enumerate(ws):
            for f, a in _fields(w, prec, 90 + s).items():
                g.set_field(s, f, a)
        g.step(3)
        g.get_field(0, "v1")  # back to the integer time level in between
        g.step(7)
        res.append([[g.get_field(s, f) for f in ("sigma", "v1", "v3")] + [g.record(s)["_all"]] for s in range(len(ws))])
        g.close()
    for s in range(len(ws)):
        for a, b, c in zip(res[0][s], res[1][s], res[2][s]):
            assert np.array_equal(a, b), s
            assert np.abs(a - c).max() <= 1e-5 * np.abs(c).max(), s
