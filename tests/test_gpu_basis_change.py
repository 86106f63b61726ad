"""Conversion between the element basis of the interface and the library's own: the state
round trip and, on both bases, one residual, for every order and for element counts around the
conversion's tile (64 triangles, 48 tetrahedra)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# 8, 64, 66, 9728, 9856, 48, 162, 6000, 7986 elements (an entry per thread up to 38,912 rows, a row above)
MESHES = [("tri", 2, 2), ("tri", 8, 4), ("tri", 11, 3), ("tri", 76, 64), ("tri", 77, 64),
          ("tet", 2, 0), ("tet", 3, 0), ("tet", 10, 0), ("tet", 11, 0)]


def mesh_of(kind, nx, ny):
    return W.bump_channel(nx, ny, 0.15, 1) if kind == "tri" else W.periodic_cube_kuhn(nx, 1.0, 0.1, 5, periodic=False)


@pytest.mark.parametrize("kind,nx,ny", MESHES)
@pytest.mark.parametrize("p", [0, 1, 2, 3])
def test_round_trip_and_norms(kind, nx, ny, p):
    import torch
    from paper_1801_06300_gb300 import capi
    if kind == "tet" and p == 3:
        pytest.skip("tetrahedra up to p = 2")
    capi.load()
    mesh, free = mesh_of(kind, nx, ny), W.Freestream()
    rng = np.random.default_rng(p)
    for prec in (capi.PCEXP_FP64, capi.PCEXP_FP32_MIXED):
        ctx = capi.Context(mesh, p, free, prec, m_max=2)
        u = rng.standard_normal(ctx.K)
        ctx.set_state(u)
        # two orthogonal blocks of at most 6 functions: a few rounding errors per entry
        assert np.abs(ctx.get_state() - u).max() <= 1e-14 * np.abs(u).max() * 6
        dev = torch.tensor(u, device="cuda")
        ctx.set_state(dev)
        assert np.abs(ctx.get_state(torch.empty_like(dev)).cpu().numpy() - u).max() <= 1e-14 * np.abs(u).max() * 6
        ctx.close()
    # the internal coefficients: same norm per element and variable (the change is orthogonal)
    a = capi.Context(mesh, p, free, capi.PCEXP_FP64, m_max=2)
    b = capi.Context(mesh, p, free, capi.PCEXP_FP64, m_max=2, basis_io=capi.PCEXP_BASIS_INTERNAL)
    prm = [0.05, 0.5, 0.5, 0.0]
    for c in (a, b):
        c.project_state(capi.PCEXP_PROJ_VORTEX, prm)
    ua, ub = a.get_state(), b.get_state()
    na, nb = (np.linalg.norm(x.reshape(-1, a.nb), axis=1) for x in (ua, ub))
    assert np.abs(na - nb).max() <= 1e-13 * na.max()
    ra, rb = a.residual(ua), b.residual(ub)
    na, nb = (np.linalg.norm(x.reshape(-1, a.nb), axis=1) for x in (ra, rb))
    assert np.abs(na - nb).max() <= 1e-11 * max(1.0, na.max())
    a.close()
    b.close()


def test_internal_basis_mixed_state_reaches_the_fp32_copy():
    """With the internal basis at the interface the FP32-mixed step still starts from the set state."""
    from paper_1801_06300_gb300 import capi
    capi.load()
    mesh, free = W.periodic_square(6, 10.0, 0.1, 3), W.Freestream(mach=0.5, alpha_deg=45.0)
    out = []
    for basis in (capi.PCEXP_BASIS_PAPER, capi.PCEXP_BASIS_INTERNAL):
        ctx = capi.Context(mesh, 2, free, capi.PCEXP_FP32_MIXED, m_max=6, basis_io=basis)
        ctx.project_state(capi.PCEXP_PROJ_VORTEX, [5.0, 5.0, 5.0, 10.0])
        u = ctx.get_state()
        ctx.project_state(capi.PCEXP_PROJ_FREESTREAM)
        ctx.set_state(u)
        ctx.step(capi.PCEXP_SCHEME_EXP1, capi.PCEXP_DT_GLOBAL_CFL, 2.0, 6)
        out.append(np.linalg.norm(ctx.get_state().reshape(-1, ctx.nb), axis=1))
        ctx.close()
    assert np.abs(out[0] - out[1]).max() <= 2e-6 * out[0].max()
