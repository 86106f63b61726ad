"""Gram-Schmidt columns of the Krylov process: the one-launch columns of short vectors and the
separate passes of longer ones and of partitions, for every number of columns and vector lengths
below one row per block, around the tiles and around the limit between the two; breakdown and
non-finite input."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "K72": lambda: (W.periodic_square(3, 10.0, 0.1, 3), 0),
    "K600": lambda: (W.periodic_square(5, 10.0, 0.1, 3), 1),
    "K13824": lambda: (W.periodic_square(24, 10.0, 0.1, 3), 1),
    "K414720": lambda: (W.periodic_square(72, 10.0, 0.1, 3), 3),
    "K960000": lambda: (W.periodic_cube_kuhn(20, 10.0, 0.1, 5, periodic=False), 1),
    # on 152 SMs: 31.2 and 32.4 KB (FP32), 99 and 101 KB (FP64) of rows per block
    "K1213488": lambda: (W.periodic_square(159, 10.0, 0.1, 3), 2),
    "K1259712": lambda: (W.periodic_square(162, 10.0, 0.1, 3), 2),
    "K1920000": lambda: (W.periodic_square(200, 10.0, 0.1, 3), 2),
    "K1958592": lambda: (W.periodic_square(202, 10.0, 0.1, 3), 2),
}
FORMS = {"selective": ("FP32_MIXED", "SELECTIVE"), "always": ("FP32_MIXED", "ALWAYS"), "fp64": ("FP64", "AUTO")}


@pytest.fixture(scope="module")
def capi():
    from paper_1801_06300_gb300 import capi as c
    c.load()
    return c


def start(ctx):
    u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb)
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(3, u.shape)).reshape(-1)
    return u, W.random_coeffs(4, u.shape)


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("form", list(FORMS))
def test_columns(capi, name, form):
    K = int(name[1:])
    if (K > 1_500_000) != (form == "fp64") and K > 500_000:
        pytest.skip("the other form's limit")
    mesh, p = MESHES[name]()
    prec, reorth = FORMS[form]
    m = 31 if K < 1_000_000 else 26 if form != "fp64" else 9
    ctx = capi.Context(mesh, p, W.Freestream(0.45, 20.0), getattr(capi, f"PCEXP_{prec}"), m_max=m,
                       reorth=getattr(capi, f"PCEXP_REORTH_{reorth}"))
    assert ctx.K == K
    u, b = start(ctx)
    V, H, k, beta = ctx.arnoldi(u, b, m)
    assert k == m
    # orthonormality and the relation at the form's rounding (its J v is computed again here, in
    # the same arithmetic): FP32 1e-5 and 2e-5; FP64 by the ratio of the unit roundoffs, 2^-29
    orth, relation = (1e-5, 2e-5) if form != "fp64" else (1e-13, 1e-13)
    assert np.abs(V @ V.T - np.eye(m + 1)).max() <= orth
    for j in range(m):
        jv = ctx.jvp(u, V[j])
        assert np.linalg.norm(H[: j + 2, j] @ V[: j + 2] - jv) <= relation * np.linalg.norm(jv), j
    ctx.close()


@pytest.mark.parametrize("name", ["K600", "K13824"])
@pytest.mark.parametrize("form", list(FORMS))
def test_one_launch_against_separate_passes(capi, name, form):
    mesh, p = MESHES[name]()
    prec, reorth = (getattr(capi, f"PCEXP_{FORMS[form][0]}"), getattr(capi, f"PCEXP_REORTH_{FORMS[form][1]}"))
    free = W.Freestream(0.45, 20.0)
    one = capi.Context(mesh, p, free, prec, m_max=31, reorth=reorth)
    grp = capi.Group(mesh, capi.partition(mesh, 2), p, free, prec, m_max=31, reorth=reorth)
    u, b = start(one)
    _, H, k, beta = one.arnoldi(u, b, 31)
    Hg, kg, bg = grp.arnoldi(u, b, 31)
    assert k == kg == 31
    # the first columns (rounding grows along a Krylov basis): sums in another order
    tol = 1e-12 if form == "fp64" else 1e-4
    assert abs(beta - bg) <= 1e-6 * bg
    assert np.linalg.norm(H[:6, :5] - Hg[:6, :5]) <= tol * np.linalg.norm(Hg[:6, :5])
    one.close()
    grp.close()


@pytest.mark.parametrize("form", list(FORMS))
def test_breakdown_and_nonfinite(capi, form):
    mesh = W.bump_channel(1, 1, 0.0, 1)  # 2 triangles at p = 0: K = 8, the space ends by column 8
    prec, reorth = FORMS[form]
    ctx = capi.Context(mesh, 0, W.Freestream(0.45, 0.0), getattr(capi, f"PCEXP_{prec}"), m_max=20,
                       eta=1e-5 if form != "fp64" else 1e-12, reorth=getattr(capi, f"PCEXP_REORTH_{reorth}"))
    u, b = start(ctx)
    V, H, k, beta = ctx.arnoldi(u, b, 20)
    assert 1 <= k <= 8
    again = ctx.arnoldi(u, b, 20)
    assert again[2] == k and np.array_equal(again[1], H)
    bad = b.copy()
    bad[3] = np.nan
    with pytest.raises(capi.PcexpError):
        ctx.arnoldi(u, bad, 20)
    after = ctx.arnoldi(u, b, 20)
    assert after[2] == k and np.array_equal(after[1], H)
    ctx.close()
