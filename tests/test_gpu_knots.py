"""Lines with knots of their own at the edges of the line solver's shapes: rows and columns of one, four and eight lines
per block, one segment of 8 positions and many, short patches, lines that no block holds (the
thread-per-patch kernel).  Oracle: B-spline collocation on the same knots; tolerances of the other knot tests."""
import numpy as np
import pytest

from oracle import nonuniform as nu

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-5}


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as ge

    ge.build()
    import paper_2301_05127_gb300 as p

    return p


def _knots(n, seed):
    h = np.exp(np.random.default_rng(seed).uniform(0.0, np.log(2.0), size=n))
    return np.concatenate([[0.0], np.cumsum(h)])


# n, p, n_nb along the axis with knots; points of the other axis
LINES = [(9, 3, 2, 9), (6, 2, 3, 40), (8, 1, 8, 700), (639, 9, 20, 33), (640, 8, 16, 19), (2559, 3, 16, 17),
         (2560, 5, 16, 18), (5120, 4, 10, 11)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("case", range(len(LINES)))
def test_knot_lines(pkg, prec, case):
    n, p, n_nb, other = LINES[case]
    x = _knots(n, case)
    for axis in (0, 1):
        nn, pp = ((n, other - 1), (p, 1)) if axis == 0 else ((other - 1, n), (1, p))
        g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[prec], n_nb, nn, pp, (1.0, 1.0), 1e-3)])
        g.set_coordinates(0, axis, x)
        f = np.random.default_rng(3).standard_normal(g.shape()).astype(g.dtype)
        ref = nu.derivative(f.astype(np.float64), axis, x, p, n_nb)
        got = g.derivative(0, axis, f)
        assert np.abs(got - ref).max() <= TOL[prec] * np.abs(ref).max(), axis
        g.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32_kahan"])
@pytest.mark.parametrize("layer", [0, 6])
def test_steps_of_one_call_equal_single_steps(pkg, prec, layer):
    """Inside one call the velocity updates at a step's end and the next one's start are one pass; with velocity
    receivers they are not.  Fields and traces have the same bits either way."""
    n, h = (48, 72), 10.0
    out = []
    for mode in range(3):
        g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[prec], 12, n, (2, 3), (h, h), 5e-4)])
        for a in (0, 1):
            g.set_coordinates(0, a, h * _knots(n[a], a))
        rho = 1000.0 + 50.0 * np.random.default_rng(1).random(g.shape())
        g.set_model(0, np.full(g.shape(), 2000.0), None, rho)
        if layer:
            g.set_pml(0, layer)
        g.set_source(0, [20, 0, 30], pkg.LOSS_SRC_PRESSURE, 1.0, 20.0, 0.005)
        rec = np.arange(0, 49 * 73, 37)
        g.set_receivers(0, "sigma", rec)
        if mode == 2:
            g.set_receivers(0, "v1", rec)
        if mode == 1:
            for _ in range(12):
                g.step(1)
        else:
            g.step(12)
        out.append([g.get_field(0, f) for f in ("sigma", "v1", "v3")] + [g.record(0)["_all"]])
        g.close()
    assert np.abs(out[0][0]).max() > 0 and np.abs(out[0][3]).max() > 0
    for a, b in zip(out[0][:3], out[1][:3]):
        assert np.array_equal(a, b)
    for a, b in zip(out[0][:3], out[2][:3]):
        assert np.array_equal(a, b)
    assert np.array_equal(out[0][3], out[1][3])
