"""The Krylov process's J v on tetrahedra, FP32 from the stored face records and FP64 from the stored
blocks, against the FP64 J v that stores nothing: faces inside and on the boundary, sub- and
supersonic (every sign of the three wave speeds), in a rotating frame, face-point counts around the
launch's block of 256."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,periodic", [(1, False), (2, False), (3, False), (3, True), (4, True)])
@pytest.mark.parametrize("p", [0, 1, 2])
@pytest.mark.parametrize("mach,omega", [(0.45, None), (2.0, None), (0.45, (0.3, -0.2, 0.5))])
def test_stored_linearisation_against_tangent(n, periodic, p, mach, omega):
    from paper_1801_06300_gb300 import capi
    if periodic and omega is not None:
        pytest.skip("a rotating frame has no translational periodicity")
    mesh = W.periodic_cube_kuhn(n, 2.0, 0.1, 5, periodic=periodic)
    if omega is not None:
        mesh.btags[:] = W.BC_SLIP_WALL
    capi.load()
    free = W.Freestream(mach=mach, alpha_deg=25.0)
    want = None
    # FP64: sums of about 50 terms in another order.  FP32: a chain of about 400 roundings of 6e-8
    # with partial cancellation between the flux's terms
    for prec, tol in ((capi.PCEXP_FP64, 1e-12), (capi.PCEXP_FP32_MIXED, 3e-5)):
        ctx = capi.Context(mesh, p, free, prec, m_max=2, omega=omega)
        if want is None:
            u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb)
            # rounded to FP32, so that both forms linearise at the same state (no branch of |x| differs)
            u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(7 + p, u.shape)).astype(np.float32).astype(np.float64)
            u = u.reshape(-1)
            v = W.random_coeffs(9, u.shape).astype(np.float32).astype(np.float64)
            want = ctx.jvp(u, v)
        V, H, k, beta = ctx.arnoldi(u, v, 1)
        got = beta * (H[0, 0] * V[0] + H[1, 0] * V[1])
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
        ctx.close()
