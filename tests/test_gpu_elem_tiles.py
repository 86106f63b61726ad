"""R(u), J(u) v and the Krylov path's J v against the oracle for element counts around the element
kernel's 32-element tile, every order, dimension and precision form, and in a rotating frame."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "tri2": lambda: (W.bump_channel(1, 1, 0.0, 1), None),
    "tri32": lambda: (W.bump_channel(8, 2, 0.15, 1), None),
    "tri66": lambda: (W.bump_channel(11, 3, 0.15, 1), None),
    "per50": lambda: (W.periodic_square(5, 10.0, 0.1, 3), None),
    "tet6": lambda: (W.periodic_cube_kuhn(1, 1.0, 0.0, 5, periodic=False), None),
    "tet48": lambda: (W.periodic_cube_kuhn(2, 1.0, 0.1, 5, periodic=False), None),
    "pertet162": lambda: (W.periodic_cube_kuhn(3, 10.0, 0.1, 5), None),
    "rot66": lambda: (W.bump_channel(11, 3, 0.15, 1), (0.0, 0.0, 0.3)),
    "rottet48": lambda: (W.periodic_cube_kuhn(2, 1.0, 0.1, 5, periodic=False), (0.2, -0.1, 0.3)),
}


@pytest.mark.parametrize("kind", list(MESHES))
@pytest.mark.parametrize("p", [0, 1, 2, 3])
def test_operator_against_oracle(kind, p):
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
    rng = np.random.default_rng(p)
    u = dg.project(lambda x: np.broadcast_to(dg.freestream_state(), x.shape[:-1] + (dg.nv,))).reshape(-1)
    u = u + 0.02 * np.abs(u).max() * rng.uniform(-1, 1, u.size)
    v = rng.standard_normal(u.size)
    R, Jv = dg.residual(u).reshape(-1), dg.jvp(u, v).reshape(-1)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)  # noqa: E731
    # perturbations of 2% in random coefficients: R is not a small difference of large terms, so
    # its relative error is a modest multiple of the form's unit roundoff
    for prec, tol in ((capi.PCEXP_FP64, 1e-12), (capi.PCEXP_FP32_MIXED, 3e-5)):
        ctx = capi.Context(mesh, p, free, prec, m_max=2, omega=omega)
        assert rel(ctx.residual(u), R) <= tol
        assert rel(ctx.jvp(u, v), Jv) <= tol
        V, H, k, beta = ctx.arnoldi(u, v, 1)
        w = beta * (H[0, 0] * V[0] + H[1, 0] * V[1])  # J v from the Krylov path
        assert rel(w, Jv) <= tol
        ctx.close()
