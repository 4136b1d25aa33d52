"""Which kernels a call takes, and what must not depend on it: handles whose shots differ in kind, explicit launch shapes,
the autotuner, and the limit of the bounded waits."""
import dataclasses
import os
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from oracle.wave import Simulation  # noqa: E402
from synth import acoustic2d_small, elastic3d_homogeneous  # noqa: E402
from synth.workloads import random_field  # noqa: E402

pytestmark = pytest.mark.gpu
FIELDS = ("sigma", "v1", "v3")


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as ge

    ge.build()
    import paper_2301_05127_gb300 as p

    return p


def _shot(n, p, n_nb, prec, seed):
    """A 2-D shot with a smooth model, a layer, and receivers of every field inside and outside the layer."""
    shape = tuple(k + 1 for k in n)
    vp = 2000.0 * (1.0 + 0.05 * random_field(shape, seed, 4.0))
    rec = np.concatenate([np.arange(shape[1]) + 3 * shape[1], np.arange(0, int(np.prod(shape)), 97)])
    w = acoustic2d_small(n=32, p=1, n_nb=n_nb, steps=10, pml_width=9)
    return dataclasses.replace(w, n=n, p=p, precision=prec, dt=0.4 * 10.0 / vp.max(),
                               model_fn=lambda: (vp, None, np.full(shape, 1000.0)), src_index=(n[0] // 2, n[1] // 2),
                               f0=40.0, t0=0.002, amp=1e4, receivers={f: rec for f in FIELDS})


def _run(pkg, ws, batched=True, graph=0, wait=None, chunks=(3, 7), seeds=None):
    """(per shot: fields and traces; launches by kernel name in the last chunk of steps) of a run from smooth fields."""
    g = pkg.Grid.from_workloads(ws)
    g.set_schedule(batched, graph)
    if wait is not None:
        g.set_wait_limit(wait)
    for s, w in enumerate(ws):
        for k, f in enumerate(FIELDS):
            a = random_field(w.shape, 70 + 3 * (seeds[s] if seeds else s) + k, 4.0) * (1.0 if f == "sigma" else 5e-7)
            g.set_field(s, f, a.astype(g.dtype))
    for c in chunks:
        g.profile(False)  # the launches of the last chunk, without those of the staggered start
        g.step(c)
    counts = {k: g.profile_read(k)[1] for k in ("acoustic_x", "acoustic_z", "acoustic_z2", "clock")}
    out = [[g.get_field(s, f) for f in FIELDS] + [g.record(s)["_all"]] for s in range(len(ws))]
    g.close()
    return out, counts


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("graph", [0, 3])
def test_mixed_fp64_handle_stays_batched(pkg, graph):
    """Shots on the engines and a shot whose patches are too short for them: one set of launches per step for each kind,
    replayed from a graph, with the fields and traces of the per-shot schedule, against the oracle."""
    geoms = [((96, 128), (2, 4), 12), ((36, 36), (3, 3), 6), ((130, 264), (2, 4), 16), ((48, 60), (4, 5), 8)]
    ws = [_shot(n, p, n_nb, "fp64", 30 + k) for k, (n, p, n_nb) in enumerate(geoms)]
    ref, single = _run(pkg, ws, batched=False)
    got, counts = _run(pkg, ws, graph=graph)
    assert single["clock"] == 0 and counts["clock"] == 7  # the clock tick is the batched schedule's
    assert counts["acoustic_z2"] == 7 and counts["acoustic_z"] == 14
    for s in range(len(ws)):
        assert _same(got[s], ref[s]), s
        sim = Simulation(ws[s])
        for k, f in enumerate(FIELDS):
            sim.state[f] = random_field(ws[s].shape, 70 + 3 * s + k, 4.0) * (1.0 if f == "sigma" else 5e-7)
        sim.step(10)
        for k, f in enumerate(FIELDS):
            err = np.linalg.norm(got[s][k] - sim.state[f]) / np.linalg.norm(sim.state[f])
            assert err < 1e-12, (s, f, err)


@pytest.mark.parametrize("prec", ["fp32", "fp32_kahan"])
def test_long_rows_do_not_depend_on_other_shots(pkg, prec):
    """FP32: a shot with long rows has the same bits alone and beside shots with short rows, in both schedules and with
    graphs, whatever the (non-zero) limit of the bounded waits; the batched step has a launch for each kind of rows."""
    long_, short = ((64, 512), (2, 4), 20), ((96, 256), (3, 2), 12)
    ws = [_shot(*g, prec, 50 + k) for k, g in enumerate([long_, short, ((96, 1024), (3, 8), 12)])]
    alone, _ = _run(pkg, ws[:1], batched=False)
    ref, _ = _run(pkg, ws, batched=False)
    assert _same(ref[0], alone[0])
    for graph, wait in ((0, None), (3, None), (0, 1 << 20)):
        got, counts = _run(pkg, ws, graph=graph, wait=wait)
        assert all(_same(a, b) for a, b in zip(got, ref)), (graph, wait)
        assert counts["acoustic_x"] == 21  # sub-steps B and A of the long rows, the pipelined kernel for the others
    other, _ = _run(pkg, ws[:1], batched=False, wait=1 << 20)
    assert _same(other[0], alone[0])
    pair, _ = _run(pkg, ws[1:2], batched=False, seeds=[1])
    assert _same(pair[0], ref[1])


ELASTIC = ("v1", "v2", "v3", "s11", "s22", "s33", "s12", "s13", "s23")
SHAPED = [("acoustic", "fp64", "acoustic_x", "line"), ("acoustic", "fp64", "acoustic_z", "line"),
          ("elastic", "fp64", "elastic_y", "line"), ("elastic", "fp32", "elastic_x", "convolution_items"),
          ("elastic", "fp32_kahan", "elastic_x", "convolution_items")]


def _engine_workload(physics, prec):
    """A grid whose FP64 acoustic or elastic step runs without launch shapes by default."""
    if physics == "acoustic":
        return _shot((64, 128), (1, 2), 12, prec, 61)
    return dataclasses.replace(elastic3d_homogeneous(n=48, p=1, n_nb=8, steps=5, precision=prec, pml_width=8), receivers={}, f0=40.0,
                               t0=0.004)


def _steps(pkg, w, n, family="convolution", shapes=()):
    g = pkg.Grid.from_workloads([w])
    g.set_kernels(family)
    for kernel, threads, chunk in shapes:
        g.set_tile(kernel, threads, chunk)
    g.step(n)
    names = FIELDS if len(w.n) == 2 else ELASTIC
    out = [g.get_field(0, f) for f in names]
    z2 = g.profile_read("acoustic_z2")[1]
    g.close()
    return out, z2


@pytest.mark.parametrize("physics,prec,kernel,family", SHAPED)
def test_shape_asked_for_is_used(pkg, physics, prec, kernel, family):
    """A launch shape belongs to the kernels that hold whole lines: with one the step is theirs, bit for bit, and without
    it again the built-in choice's."""
    w = _engine_workload(physics, prec)
    plain, z2 = _steps(pkg, w, 5)
    ref, _ = _steps(pkg, w, 5, family, [(kernel, 128, 4)])
    got, got_z2 = _steps(pkg, w, 5, shapes=[(kernel, 128, 4)])
    assert np.abs(ref[0]).max() > 0 and not _same(plain, ref)  # the two families differ in rounding
    assert _same(got, ref)
    assert got_z2 == 0 and (physics == "elastic" or z2 > 0)
    back, _ = _steps(pkg, w, 5, shapes=[(kernel, 128, 4), (kernel, 0, 0)])
    assert _same(back, plain)


@pytest.mark.parametrize("physics,prec", [("acoustic", "fp64"), ("elastic", "fp64"), ("elastic", "fp32_kahan")])
def test_autotune_reports_what_runs(pkg, physics, prec):
    """Steps without launch shapes: the tuner's entries are the built-in choice for all kernels or a shape for each, and
    the tuned handle runs what they say."""
    w = _engine_workload(physics, prec)
    g = pkg.Grid.from_workloads([w])
    res = g.autotune(steps=2)
    assert set(res) == ({"acoustic_x", "acoustic_z"} if physics == "acoustic" else {"elastic_x", "elastic_y", "elastic_z"})
    assert all(r["ms"] > 0 for r in res.values())
    built_in = [r["threads_per_block"] == 0 and r["chunk_log2"] == 0 for r in res.values()]
    assert all(built_in) or not any(built_in)
    g.step(5)
    got = [g.get_field(0, f) for f in (FIELDS if physics == "acoustic" else ELASTIC)]
    assert physics == "elastic" or (g.profile_read("acoustic_z2")[1] > 0) == built_in[0]
    g.close()
    ref, _ = _steps(pkg, w, 5, shapes=[(k, r["threads_per_block"], r["chunk_log2"]) for k, r in res.items()])
    assert _same(got, ref)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("axis", [0, 1])
def test_transpose_over_its_input(pkg, prec, axis):
    """Device arrays that share memory are refused, the same host array twice is not."""
    import ctypes

    import torch

    w = dataclasses.replace(_shot((64, 128), (1, 2), 12, prec, 5), receivers={})
    g = pkg.Grid.from_workloads([w])
    a = random_field(w.shape, 3, 4.0).astype(g.dtype)
    ref = g.derivative_adjoint(0, axis, a)
    f = pkg.lib().loss_derivative_adjoint
    buf = torch.zeros(3 * a.size, dtype=torch.from_numpy(a).dtype, device="cuda")
    buf[:a.size] = torch.from_numpy(a).reshape(-1).cuda()
    torch.cuda.synchronize()
    p, nb = buf.data_ptr(), a.nbytes
    for out in (p, p + nb - a.itemsize):
        assert f(g.h, 0, axis, ctypes.c_void_p(p), ctypes.c_void_p(out), pkg.LOSS_MEM_DEVICE) == pkg.LOSS_E_ARG
    assert f(g.h, 0, axis, ctypes.c_void_p(p), ctypes.c_void_p(p + nb), pkg.LOSS_MEM_DEVICE) == pkg.LOSS_OK
    g.sync()
    assert np.array_equal(buf[a.size:2 * a.size].cpu().numpy().reshape(a.shape), ref)
    b = a.copy()
    assert f(g.h, 0, axis, b.ctypes.data, b.ctypes.data, pkg.LOSS_MEM_HOST) == pkg.LOSS_OK
    assert np.array_equal(b, ref)
    g.close()


@pytest.mark.parametrize("prec", ["fp32", "fp32_kahan"])
def test_short_rows_after_the_row_engine(pkg, prec):
    """A batch whose pipelined x kernel has blocks of several warps (rows of 257 to 512 points, two groups of rows in a
    block, blocks that go from one shot to the next) and follows the row kernel's launches of the long shots."""
    sizes = [(12, 64), (4, 64), (5, 64), (7, 64), (4, 96), (9, 96), (4, 64)]
    ws = [_shot((512, k * m), (4, k), 12, prec, 80 + i) for i, (k, m) in enumerate(sizes)]
    ref, _ = _run(pkg, ws, batched=False)
    for graph in (0, 3):
        got, counts = _run(pkg, ws, graph=graph, chunks=(3, 9))
        again, _ = _run(pkg, ws, graph=graph)
        assert counts["acoustic_x"] == 27
        assert all(_same(a, b) for a, b in zip(again, ref)), graph
        assert np.isfinite(got[0][0]).all()


@pytest.mark.parametrize("physics,kernel", [("acoustic", "acoustic_z"), ("elastic", "elastic_x")])
@pytest.mark.parametrize("graph", [0, 2])
def test_shape_set_between_steps(pkg, physics, kernel, graph):
    """A launch shape set and taken back between steps moves the run to the other kernels and back: the fields stay those
    of the run without it, to the tolerance of the FP64 form."""
    w = _engine_workload(physics, "fp64")
    out = []
    for shapes in ([None] * 3, [None, (128, 4), (0, 0)]):
        g = pkg.Grid.from_workloads([w])
        g.set_schedule(True, graph)
        for s in shapes:
            if s is not None:
                g.set_tile(kernel, *s)
            g.step(4)
        out.append([g.get_field(0, f) for f in (FIELDS if physics == "acoustic" else ELASTIC)])
        g.close()
    assert not _same(*out)
    names = FIELDS if physics == "acoustic" else ELASTIC
    for f, a, b in zip(names, *out):  # against the largest field of its kind (velocities, stresses)
        scale = max(np.linalg.norm(x) for k, x in zip(names, out[0]) if k[0] == f[0])
        assert np.linalg.norm(a - b) <= 1e-12 * scale, f
