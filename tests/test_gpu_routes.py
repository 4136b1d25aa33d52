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
