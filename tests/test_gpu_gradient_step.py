"""loss_gradient's forward run against loss_step's: traces of the same model give misfit zero and gradients zero."""
import dataclasses

import numpy as np
import pytest

from synth import acoustic2d_gradient_case, elastic3d_gradient_case
from synth.workloads import random_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as ge

    ge.build()
    import paper_2301_05127_gb300 as p

    return p


def _case(kind, prec):
    """Acoustic rows of 513 points or 3-D elastic, in sizes that the column and row engines take."""
    if kind == "elastic":
        w, _ = elastic3d_gradient_case(precision=prec)
        n, p = (40, 44, 48), (1, 1, 1)
        base = (3000.0, 1730.0, 2000.0)
    else:
        w, _ = acoustic2d_gradient_case(precision=prec)
        n, p = ((48, 512), (1, 4)) if kind == "long rows" else ((48, 2310), (1, 11))
        base = (2000.0, None, 1000.0)
    shape = tuple(k + 1 for k in n)
    m = tuple(None if b is None else b * (1.0 + 0.05 * random_field(shape, 5 + i, 4.0)) for i, b in enumerate(base))
    src = tuple(k // 2 for k in n)
    plane = int(np.prod(shape[1:]))
    rec = (src[0] - 4) * plane + np.arange(0, plane, 3)
    return dataclasses.replace(w, n=n, p=p, n_nb=8, precision=prec, model_fn=lambda: m, src_index=src, dt=1e-3, f0=40.0,
                               t0=0.004, steps=12, pml_width=8, receivers={f: rec for f in w.receivers})


@pytest.mark.parametrize("family", ["convolution", "convolution_items", "line"])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_kahan"])
@pytest.mark.parametrize("kind", ["elastic", "long rows", "ragged rows"])
def test_own_traces_have_no_misfit(pkg, kind, prec, family):
    """Exactly, but for FP32 on the convolution family, whose loss_step runs on the engines and whose gradient does not:
    there the traces agree to FP32 rounding."""
    w = _case(kind, prec)
    g = pkg.Grid.from_workloads([w])
    g.set_kernels(family)
    g.step(w.steps)
    obs = g.record(0)["_all"].astype(np.float64)
    assert np.abs(obs).max() > 0
    J, grads = g.gradient(0, obs, w.steps)
    tr = g.record(0)["_all"]
    g.close()
    if prec != "fp64" and family == "convolution":
        assert np.abs(tr - obs).max() <= 1e-5 * np.abs(obs).max()
        assert J <= 0.5 * 1e-10 * obs.size * np.abs(obs).max() ** 2
        return
    assert J == 0.0 and np.array_equal(tr, obs)
    assert not any(np.any(v) for v in grads.values() if v is not None)


def test_gradient_after_a_new_model(pkg):
    """The chain rule's model follows loss_set_model, on a stream that does not wait for the legacy default stream: a
    handle's second gradient, at another model, has the bits of a fresh handle's."""
    import torch

    w = _case("long rows", "fp64")
    vp, vs, rho = w.model_fn()
    models = [(vp, vs, rho), (np.ascontiguousarray(vp[::-1]), vs, 0.97 * rho)]  # (of one largest vp: the layer's)
    st = torch.cuda.Stream()
    obs = None
    out = []
    g = pkg.Grid.from_workloads([w], stream=st)
    for m in models:
        f = pkg.Grid.from_workloads([dataclasses.replace(w, model_fn=lambda: m)], stream=st)
        if obs is None:
            f.step(w.steps)
            obs = 0.9 * f.record(0)["_all"].astype(np.float64)
        fresh = f.gradient(0, obs, w.steps)
        f.close()
        g.set_model(0, *m)
        out.append((g.gradient(0, obs, w.steps), fresh))
    g.close()
    for (J, a), (K, b) in out:
        assert J == K and J > 0
        for k in ("vp", "rho"):
            assert np.any(a[k]) and np.array_equal(a[k], b[k]), k
    assert not np.array_equal(out[0][0][1]["rho"], out[1][0][1]["rho"])
