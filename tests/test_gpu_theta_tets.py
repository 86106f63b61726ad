"""The reverse step's adjoint of (Mach number, flow angle) on tetrahedra with far-field faces and slip
walls, against central differences of the step itself at a fixed state."""
import dataclasses

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [0, 1, 2])
def test_theta_adjoint_against_differences(p):
    from paper_1801_06300_gb300 import capi
    capi.load()
    mesh = W.periodic_cube_kuhn(2, 1.0, 0.1, 5, periodic=False)
    z = mesh.coords[mesh.bfaces][:, :, 2]
    mesh.btags[(z == z[:, :1]).all(1) & ((z[:, 0] == 0.0) | (z[:, 0] == 1.0))] = W.BC_SLIP_WALL
    free = W.Freestream(mach=0.45, alpha_deg=12.0)
    ctx = capi.Context(mesh, p, free, capi.PCEXP_FP64, m_max=8)
    u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb)
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(3, u.shape)).reshape(-1)
    w = W.random_coeffs(4, u.shape)
    dt, m = 0.02, 8

    def step(**kw):
        ctx.set_physics(dataclasses.replace(free, **kw))
        ctx.set_state(u)
        ctx.step(capi.PCEXP_SCHEME_PCEXP, capi.PCEXP_DT_GIVEN, dt, m)
        return ctx.get_state()

    # central differences: truncation h^2 f''' / 6 and rounding eps |u| / h are both below 1e-8 of the
    # derivative's size
    want, size = [], []
    for name, h in (("mach", 1e-5), ("alpha_deg", 1e-3)):
        d = (step(**{name: getattr(free, name) + h}) - step(**{name: getattr(free, name) - h})) / (2 * h)
        want.append(w @ d)
        size.append(np.linalg.norm(w) * np.linalg.norm(d))
    ctx.set_physics(free)
    _, theta = ctx.step_backward(u, dt, m, w, with_theta=True)
    for k in range(2):
        assert size[k] > 0 and abs(theta[k] - want[k]) <= 1e-6 * size[k], k
    ctx.close()
