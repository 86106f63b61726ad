"""The element kernel's two forms (four lanes per element on meshes of up to 32 elements per SM, one
above) against the oracle for element counts on both sides of the limit: R(u), J(u) v and the
Krylov path's J v."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {  # limit on 152 SMs: 4864 elements
    "tri4802": lambda: (W.periodic_square(49, 10.0, 0.1, 3), None),
    "tri5000": lambda: (W.periodic_square(50, 10.0, 0.1, 3), None),
    "tet4374": lambda: (W.periodic_cube_kuhn(9, 10.0, 0.1, 5), None),
    "tet6000": lambda: (W.periodic_cube_kuhn(10, 10.0, 0.1, 5, periodic=False), None),
    "rot4860": lambda: (W.bump_channel(81, 30, 0.15, 1), (0.0, 0.0, 0.3)),
    "rot5084": lambda: (W.bump_channel(82, 31, 0.15, 1), (0.0, 0.0, 0.3)),
}


@pytest.mark.parametrize("kind", list(MESHES))
@pytest.mark.parametrize("p", [1, 2, 3])
def test_forms_against_oracle(kind, p):
    from oracle.dg import DGOracle
    from paper_1801_06300_gb300 import capi
    mesh, omega = MESHES[kind]()
    if mesh.dim == 3 and p == 3:
        pytest.skip("tetrahedra up to p = 2")
    if omega is not None:
        mesh.btags[:] = W.BC_SLIP_WALL
    capi.load()
    free = W.Freestream(mach=0.45, alpha_deg=12.0)
    dg = DGOracle(mesh, p, free, omega)
    u = dg.project(lambda x: np.broadcast_to(dg.freestream_state(), x.shape[:-1] + (dg.nv,)))
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(p, u.shape)).reshape(-1)
    v = W.random_coeffs(7, u.shape)
    R, Jv = dg.residual(u).reshape(-1), dg.jvp(u, v).reshape(-1)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    # as for the tiles: 2% in random coefficients, a modest multiple of the form's unit roundoff
    for prec, tol in ((capi.PCEXP_FP64, 1e-12), (capi.PCEXP_FP32_MIXED, 3e-5)):
        ctx = capi.Context(mesh, p, free, prec, m_max=2, omega=omega)
        assert rel(ctx.residual(u), R) <= tol
        assert rel(ctx.jvp(u, v), Jv) <= tol
        V, H, k, beta = ctx.arnoldi(u, v, 1)
        assert rel(beta * (H[0, 0] * V[0] + H[1, 0] * V[1]), Jv) <= tol
        ctx.close()
