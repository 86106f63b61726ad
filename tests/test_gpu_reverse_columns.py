"""The reverse Gram-Schmidt columns of step_backward for column counts around the warps' shares of
8 and vector lengths below, around and above one wave of 256-row tiles: the gradient's directional
derivative against central differences of the step itself."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "K72": lambda: (W.periodic_square(3, 10.0, 0.1, 3), 0),
    "K600": lambda: (W.periodic_square(5, 10.0, 0.1, 3), 1),
    "K13824": lambda: (W.periodic_square(24, 10.0, 0.1, 3), 1),
    "K81920": lambda: (W.periodic_square(32, 10.0, 0.1, 3), 3),
}


@pytest.mark.parametrize("name,m", [("K72", 8), ("K72", 17), ("K600", 1), ("K600", 9), ("K600", 30), ("K13824", 16),
                                    ("K13824", 25), ("K81920", 24), ("K81920", 31)])
def test_directional_derivative(name, m):
    from paper_1801_06300_gb300 import capi
    mesh, p = MESHES[name]()
    capi.load()
    ctx = capi.Context(mesh, p, W.Freestream(0.45, 20.0), capi.PCEXP_FP64, m_max=m)
    u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb)
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(3, u.shape)).reshape(-1)
    ctx.set_state(u)
    dt = ctx.step(capi.PCEXP_SCHEME_PCEXP, capi.PCEXP_DT_GLOBAL_CFL, 1.0, m)["dt"]
    g = W.random_coeffs(5, u.shape)
    ub = ctx.step_backward(u, dt, m, g)

    def J(x):
        ctx.set_state(x)
        ctx.step(capi.PCEXP_SCHEME_PCEXP, capi.PCEXP_DT_GIVEN, dt, m, info=False)
        return g @ ctx.get_state()

    delta = W.random_coeffs(6, u.shape) * np.abs(u)
    h = 1e-5  # truncation h^2, rounding 1e-16 / h: well below the bound
    fd = (J(u + h * delta) - J(u - h * delta)) / (2 * h)
    assert abs(ub @ delta - fd) <= 1e-5 * np.linalg.norm(ub) * np.linalg.norm(delta)
    assert abs(ub @ delta - fd) <= 1e-4 * abs(fd)
    ctx.close()
