"""The polynomial that preconditions the FP64 solves (rve_debug_chebyshev, host code of the
library; no GPU needed), run as a scalar recurrence on one eigenvalue t of D^-1 A: z(1) is
the polynomial's value and t z(1) the eigenvalue of the preconditioned operator."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def rve():
    from paper_1610_03484_gb300 import _build
    _build.build()
    import paper_1610_03484_gb300 as pkg
    pkg.load_library()
    return pkg


def preconditioned(rve, lam, ratio, t):
    w, steps = rve.chebyshev(lam, ratio)
    z = np.full_like(t, w)
    d = z.copy()
    for c1, c2 in steps.astype(np.float64):
        d = c1 * d + c2 * (1.0 - t * z)
        z = z + d
    return t * z, len(steps) + 1


@pytest.mark.parametrize("ratio", [10.0, 15.0, 36.0, 100.0, 144.0, 198.0, 250.0, 300.0, 576.0, 907.0, 1024.0, 1500.0])
def test_positive_definite_on_both_sides_of_the_estimate(rve, ratio):
    """Eigenvalues inside the interval come out within 1 / T(th / de) of 1 (T the Chebyshev
    polynomial of the degree; FP32 coefficients add about 1e-5), those up to half as large
    again above it positive."""
    lam = 2.75
    mu, degree = preconditioned(rve, lam, ratio, np.linspace(lam / ratio, lam, 2001))
    th, de = 0.5 * (lam + lam / ratio), 0.5 * (lam - lam / ratio)
    delta = 1.0 / np.cosh(degree * np.arccosh(th / de))
    assert np.abs(mu - 1.0).max() <= delta + 1e-4
    assert degree >= np.sqrt(ratio) - 1
    above, _ = preconditioned(rve, lam, ratio, np.linspace(lam, 1.5 * lam, 2001))
    below, _ = preconditioned(rve, lam, ratio, np.linspace(1e-6, lam / ratio, 2001))
    assert (above > 0).all() and (below > 0).all()


def test_arguments(rve):
    for lam, ratio in ((0.0, 10.0), (-1.0, 10.0), (1.0, 1.0), (float("nan"), 10.0)):
        with pytest.raises(rve.RveError):
            rve.chebyshev(lam, ratio)
