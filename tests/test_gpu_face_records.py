"""The FP32 J v on tetrahedra recomputes the Roe flux's derivative from stored records; compared with
the FP64 form, which multiplies stored Jacobian blocks: faces inside and on the boundary, sub- and
supersonic, in a rotating frame, face-point counts around the launch's block of 256."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,periodic", [(1, False), (2, False), (3, False), (3, True), (4, True)])
@pytest.mark.parametrize("p", [0, 1, 2])
@pytest.mark.parametrize("mach,omega", [(0.45, None), (2.0, None), (0.45, (0.3, -0.2, 0.5))])
def test_records_against_blocks(n, periodic, p, mach, omega):
    from paper_1801_06300_gb300 import capi
    if periodic and omega is not None:
        pytest.skip("a rotating frame has no translational periodicity")
    mesh = W.periodic_cube_kuhn(n, 2.0, 0.1, 5, periodic=periodic)
    if omega is not None:
        mesh.btags[:] = W.BC_SLIP_WALL
    capi.load()
    free = W.Freestream(mach=mach, alpha_deg=25.0)
    out = []
    for prec in (capi.PCEXP_FP64, capi.PCEXP_FP32_MIXED):
        ctx = capi.Context(mesh, p, free, prec, m_max=2, omega=omega)
        u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb) if prec == capi.PCEXP_FP64 else u
        if prec == capi.PCEXP_FP64:
            # rounded to FP32, so that both forms linearise at the same state (no branch of |x| differs)
            u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(7 + p, u.shape)).astype(np.float32).astype(np.float64)
            v = W.random_coeffs(9, u.shape).astype(np.float32).astype(np.float64).reshape(-1)
        out.append(ctx.jvp(u.reshape(-1), v))
        ctx.close()
    # a chain of about 400 roundings of 6e-8 with partial cancellation between the flux's terms
    assert np.linalg.norm(out[1] - out[0]) <= 3e-5 * np.linalg.norm(out[0])
