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


@pytest.mark.parametrize("axis", [0, 1])
def test_left_out_weights_stay_below_the_last_digit(pkg, axis):
    """FP64: a sample beyond the halo of a junction (n_nb < m <= 32) has no weight there, so its derivative at the
    junction is 0, and so is the transpose at the sample.  The convolution's own term cancels against the correction's
    weight: what is left is at most the sum of the weights left out, 2^-58, and the term beyond 32 positions, A |r|^32."""
    n, p, n_nb = 128, 2, 12
    g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.LOSS_FP64, n_nb, (n, n), (p, p), (1.0, 1.0), 1e-3)])
    f = np.zeros(g.shape())
    t = np.zeros(g.shape())
    dist = [(k, m) for k, m in enumerate([s * m for m in range(n_nb + 1, 33) for s in (1, -1)])]
    for k, m in dist:
        f[k, 64 + m] = 1.0
        t[k, 64] = 1.0
    if axis == 0:
        f, t = f.T.copy(), t.T.copy()
    d = g.derivative(0, axis, f)
    a = g.derivative_adjoint(0, axis, t)
    if axis == 0:
        d, a = d.T, a.T
    g.close()
    bound = 3.0 * (2.0 ** -58 + A * 0.26794919243112270647 ** 32)
    assert max(abs(d[k, 64]) for k, _ in dist) <= bound
    assert max(abs(a[k, 64 + m]) for k, m in dist) <= bound


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_axes_of_many_patches(pkg, prec):
    """120 patches: the derivative's tables still fit the static array of the variant without allocations, the transpose's
    are larger.  Against dense matrices of the oracle, and the same bits from the variant."""
    import ctypes

    import torch

    from oracle import spline

    n, p, n_nb = 3360, 120, 20
    tol = 1e-12 if prec == "fp64" else 2e-5
    d = pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[prec], n_nb, (n, 20), (p, 1), (1.0, 1.0), 1e-3)
    g = pkg.Grid([d])
    f = np.random.default_rng(4).standard_normal(g.shape()).astype(g.dtype)
    D = spline.derivative(np.eye(n + 1), 0, n, p, 1.0, n_nb)
    for op, ref in ((g.derivative, D @ f), (g.derivative_adjoint, D.T @ f)):
        assert np.abs(op(0, 0, f) - ref).max() < tol * np.abs(ref).max()
    x = torch.from_numpy(f).cuda()
    out = torch.empty_like(x)
    st = pkg.lib().loss_derivative_noalloc(ctypes.byref(d), 0, x.data_ptr(), out.data_ptr(),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == pkg.LOSS_OK
    assert np.array_equal(out.cpu().numpy(), g.derivative(0, 0, f))
    g.close()


@pytest.mark.parametrize("prec", ["fp32", "fp32_kahan"])
def test_density_array_has_no_common_error(pkg, prec):
    """v1 of one step from a pressure field, the density an array and the density a constant of the same value: both round
    point by point (about 2 u each, u = 2^-24, over 33000 points: 1e-9 of the common factor), and no factor is common to
    all points.  dt is one at which the FP32 product of step length and derivative scale is far from the exact one."""
    n, p = (64, 512), (1, 4)
    scale = A * 3.0 / 10.0

    def bias(dt):
        s, c = np.float32(scale), np.float32(dt)
        return abs(float(np.float32(s * c)) / (float(s) * float(c)) - 1.0)

    dt = max((1e-3 * (1.0 + k / 64.0) for k in range(64)), key=bias)
    assert bias(dt) > 3e-8
    rng = np.random.default_rng(2)
    out = []
    for array in (False, True):
        g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[prec], 12, n, p, (10.0, 10.0), dt)])
        rho = np.full(g.shape(), 1024.0)
        if array:
            rho[0, 0] = 512.0  # 1 / rho exact in FP32
        g.set_model(0, np.full(g.shape(), 1e-6), None, rho)  # the pressure does not move
        if not out:
            f = rng.standard_normal(g.shape()).astype(np.float32)
        g.set_field(0, "sigma", f)
        g.step(1)
        out.append(g.get_field(0, "v1").astype(np.float64)[1:])
        g.close()
    c, a = out
    assert abs(np.sum((a - c) * c) / np.sum(c * c)) <= 5e-9


@pytest.mark.parametrize("prec", ["fp32", "fp32_kahan"])
def test_row_engine_has_no_common_error(pkg, prec):
    """v1 of one step from smooth pressure rows against the FP64 handle's.  A point's error is a few u times |f| over the
    difference 0.2 |f| of its sums, about 5 u = 3e-7 at 40 points a wavelength, independent from point to point (rows of
    random phase and amplitude): 4e-10 of the common factor over 525000 points.  Three times that is allowed; r rounded to
    FP32 alone would leave 2.0e-9."""
    n, p = (512, 1024), (4, 8)
    rng = np.random.default_rng(11)
    x = np.arange(n[1] + 1)
    f = (rng.uniform(0.5, 2.0, (n[0] + 1, 1)) * np.sin(2 * np.pi * x / 40.0 + rng.uniform(0, 6.28, (n[0] + 1, 1))))
    f = f.astype(np.float32)
    out = {}
    for q in ("fp64", prec):
        g = pkg.Grid([pkg.make_desc(2, pkg.LOSS_ACOUSTIC, pkg.PRECISIONS[q], 20, n, p, (10.0, 10.0), 1e-3)])
        g.set_model(0, np.full(g.shape(), 1e-6), None, np.full(g.shape(), 1024.0))  # the pressure does not move
        g.set_field(0, "sigma", f.astype(g.dtype))
        g.step(1)
        out[q] = g.get_field(0, "v1").astype(np.float64)
        g.close()
    c, a = out["fp64"], out[prec]
    assert abs(np.sum((a - c) * c) / np.sum(c * c)) <= 1.2e-9
