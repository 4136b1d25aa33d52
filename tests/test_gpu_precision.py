"""Precision of the junction corrections and coefficients on the column and row engines: weights that are left out, the
transpose at small halo widths, and the coefficient of the velocity update with a density array."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
A = (1.0 - (2.0 - 3.0 ** 0.5) ** 2) / (2.0 * 3.0 ** 0.5)  # e_i = A (R_i - L_i), derivative 3 e / h


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as ge

    ge.build()
    import paper_2301_05127_gb300 as p

    return p


@pytest.mark.parametrize("n_nb", [1, 2, 5])
@pytest.mark.parametrize("axis", [0, 1])
def test_fp32_transpose_at_small_halos(pkg, axis, n_nb):
    """The corrections are largest here (0.07 of a sample at n_nb = 1).  Against the same operator in FP64: with samples
    of at most G, the two recursions round to 2 u G / (1 - |r|)^2 together, the difference, the correction and the scale
    to 2 u G each (u = 2^-24)."""
    n, p, h = (192, 264), (2, 3), 1.0
    out = []
    x = np.random.default_rng(n_nb).uniform(-1.0, 1.0, (193, 265)).astype(np.float32)
    for prec in (pkg.LOSS_FP32, pkg.LOSS_FP64):
        g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, prec, n_nb, n, p, (h, h), 1e-3)])
        out.append(g.derivative_adjoint(0, axis, x.astype(g.dtype)).astype(np.float64))
        g.close()
    u, q = 2.0 ** -24, 1.0 / (1.0 - 0.268) ** 2
    # line ends: the reflection's terms, 2 / (1 - |r|) of the end sums
    ends = np.ones(x.shape[axis])
    ends[[0, -1]] = 3.0
    tol = 3.0 * A * u * (2.0 * q + 6.0) * ends
    tol = tol[:, None] if axis == 0 else tol[None, :]
    assert (np.abs(out[0] - out[1]) <= tol).all()
    assert np.sqrt(np.mean((out[0] - out[1]) ** 2)) <= 0.25 * 3.0 * A * u * (2.0 * q + 6.0)
