"""phi_1 / phi_2 of small matrices and its adjoint over the sizes and norms where the scaling and
squaring changes course (no squaring, one, many; rows that do not divide among the cluster)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import workloads as W
    from paper_1801_06300_gb300 import capi
    capi.load()
    c = capi.Context(W.periodic_square(4, 1.0), 0, W.Freestream(), capi.PCEXP_FP64, m_max=4)
    yield c
    c.close()


def hessenberg(k, scale):
    rng = np.random.default_rng(100 * k + 7)
    return np.triu(rng.standard_normal((k, k)), -1) * scale / np.sqrt(k) - scale * np.eye(k)


# the squarings multiply the rounding of one product (k + 2 terms) by at most 2^s for a contraction:
# (k + 2) 2^s eps with 2^s <= 4 ||dt H||_1 stays below 1e-12 up to norms of about 30
@pytest.mark.parametrize("k", [1, 2, 5, 6, 7, 8, 14, 15, 31, 32])
@pytest.mark.parametrize("scale", [1e-9, 0.05, 0.3, 1.0, 8.0])
def test_phi_against_extended_precision(ctx, k, scale):
    from oracle.krylov import phi_e1
    H = hessenberg(k, scale)
    p1, p2 = ctx.phi(H, 0.7)
    o1, o2 = phi_e1(H, 0.7)
    assert np.linalg.norm(p1 - o1) <= 1e-12 * np.linalg.norm(o1)
    assert np.linalg.norm(p2 - o2) <= 1e-12 * np.linalg.norm(o2)


# y = phi_1(dt H) e_1: <ybar, dy> = <Hbar, dH> with dy from a complex step of the oracle
@pytest.mark.parametrize("k", [1, 6, 15, 32])
@pytest.mark.parametrize("scale", [1e-9, 0.3, 8.0])
def test_phi_adjoint_against_complex_step(ctx, k, scale):
    from oracle.krylov import phi_e1
    rng = np.random.default_rng(k)
    H, dH, yb = hessenberg(k, scale), rng.standard_normal((k, k)), rng.standard_normal(k)
    Hb = ctx.phi_adjoint(H, 0.7, yb)
    dy = phi_e1(H + 1e-30j * dH, 0.7)[0].imag / 1e-30
    size = np.linalg.norm(Hb) * np.linalg.norm(dH)
    assert abs(np.sum(Hb * dH) - yb @ dy) <= 1e-11 * size


def test_phi_non_finite_is_reported(ctx):
    from paper_1801_06300_gb300 import capi
    for bad in (np.nan, np.inf):
        H = hessenberg(6, 1.0)
        H[2, 3] = bad
        with pytest.raises(capi.PcexpError) as e:
            ctx.phi(H, 0.7)
        assert e.value.code == capi.PCEXP_ERR_NONFINITE
