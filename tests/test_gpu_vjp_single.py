"""J(u)^T w without stored Jacobians: the transpose identity <w, J v> = <J^T w, v> on every order,
boundary type and precision form, in a rotating frame too, for element counts that leave ragged
tiles; and the face blocks of the Krylov path against the matrix-free J v."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def mesh_of(kind):
    free = W.Freestream(mach=0.45, alpha_deg=12.0)
    if kind == "bump":
        return W.bump_channel(9, 5, 0.15, 1), free, None
    if kind == "square":
        return W.periodic_square(5, 10.0, 0.1, 3), free, None
    mesh = W.periodic_cube_kuhn(3, 1.0, 0.1, 5, periodic=False)
    if kind == "box":
        return mesh, free, None
    mesh.btags[:] = W.BC_SLIP_WALL  # walled box in a rotating frame
    return mesh, free, (0.2, -0.1, 0.3)


@pytest.mark.parametrize("kind", ["bump", "square", "box", "rotating"])
@pytest.mark.parametrize("p", [0, 1, 2, 3])
def test_transpose_identity(kind, p):
    from paper_1801_06300_gb300 import capi
    mesh, free, omega = mesh_of(kind)
    if mesh.dim == 3 and p == 3:
        pytest.skip("tetrahedra up to p = 2")
    capi.load()
    rng = np.random.default_rng(10 * p)
    # one J v is a sum of a few hundred terms: 1e-13 in FP64 and 1e-5 in FP32 of the factors' sizes
    for prec, tol in ((capi.PCEXP_FP64, 1e-13), (capi.PCEXP_FP32_MIXED, 1e-5)):
        ctx = capi.Context(mesh, p, free, prec, m_max=2, omega=omega)
        ctx.project_state(capi.PCEXP_PROJ_FREESTREAM)
        u = ctx.get_state()
        u = u + 0.02 * np.abs(u).max() * rng.uniform(-1, 1, u.size)
        v, w = rng.standard_normal((2, u.size))
        Jv, JTw = ctx.jvp(u, v), ctx.vjp(u, w)
        size = np.linalg.norm(Jv) * np.linalg.norm(w) + np.linalg.norm(JTw) * np.linalg.norm(v)
        assert abs(w @ Jv - JTw @ v) <= tol * size
        # the Krylov path: h_11 = <v, J v> / <v, v> from the stored point Jacobians
        _, H, k, beta = ctx.arnoldi(u, v, 1)
        assert abs(H[0, 0] - v @ Jv / (v @ v)) <= tol * np.linalg.norm(Jv) / np.linalg.norm(v)
        ctx.close()
