"""phi_1 / phi_2 of matrices of large norm (many squarings), as a stiff step's Hessenberg matrix at a
large CFL number: contractions with real and with oscillating spectra."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def contraction(k, scale, skew):
    """Tridiagonal, symmetric part negative semi-definite, ||H||_1 about scale."""
    lap = (np.diag(-2.0 * np.ones(k)) + np.diag(np.ones(k - 1), 1) + np.diag(np.ones(k - 1), -1)) / 4.0
    rot = (np.diag(np.ones(k - 1), -1) - np.diag(np.ones(k - 1), 1)) / 2.0
    return scale * ((1.0 - skew) * lap + skew * rot)


# s squarings of a contraction multiply the rounding of one product (k + 2 terms, unit roundoff
# 1.1e-16) by at most 2^s <= 4 max(||dt H||_1, 1)
@pytest.mark.parametrize("k", [2, 9, 16, 30, 32])
@pytest.mark.parametrize("scale", [30.0, 1e3, 3e4])
@pytest.mark.parametrize("skew", [0.0, 0.5, 1.0])
def test_phi_of_stiff_contractions(k, scale, skew):
    import workloads as W
    from oracle.krylov import phi_e1
    from paper_1801_06300_gb300 import capi
    capi.load()
    ctx = capi.Context(W.periodic_square(4, 1.0), 0, W.Freestream(), capi.PCEXP_FP64, m_max=4)
    H, dt = contraction(k, scale, skew), 0.7
    norm = max(np.abs(dt * H).sum(0).max(), 1.0)
    tol = (k + 2) * 4.0 * norm * 1.2e-16
    # against the vectors' natural size: |phi_j e_1| of a contraction is at most 1
    for got, want in zip(ctx.phi(H, dt), phi_e1(H, dt)):
        assert np.linalg.norm(got - want) <= tol
    ctx.close()
