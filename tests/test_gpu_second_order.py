"""Second-order adjoint (d(J(u) v)/du)^T w and the reverse step's free-stream adjoint, on every order
and boundary type, against derivatives of the oracle's J v taken by a complex step."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def mesh_of(kind):
    free = W.Freestream(mach=0.45, alpha_deg=12.0)
    if kind == "bump":   # walls and far field
        return W.bump_channel(7, 3, 0.15, 1), free
    if kind == "square":  # periodic
        return W.periodic_square(4, 10.0, 0.1, 3), free
    mesh = W.periodic_cube_kuhn(2, 1.0, 0.1, 5, periodic=False)  # far field, two walls
    z = mesh.coords[mesh.bfaces][:, :, 2]
    mesh.btags[(z == z[:, :1]).all(1) & ((z[:, 0] == 0.0) | (z[:, 0] == 1.0))] = W.BC_SLIP_WALL
    return mesh, free


# two independent evaluations in FP64 of sums of at most ~50 terms through a flux and its second
# derivative: 1e-10 of the result's size is far above their rounding and far below any wrong term
@pytest.mark.parametrize("kind,p", [("bump", 0), ("bump", 1), ("bump", 2), ("bump", 3), ("square", 2), ("box", 0),
                                    ("box", 1), ("box", 2)])
def test_second_order_against_complex_step(kind, p):
    from oracle.dg import DGOracle
    from paper_1801_06300_gb300 import capi
    capi.load()
    mesh, free = mesh_of(kind)
    dg = DGOracle(mesh, p, free)
    rng = np.random.default_rng(p)
    u = dg.project(lambda x: np.broadcast_to(dg.freestream_state(), x.shape[:-1] + (dg.nv,))).reshape(-1)
    u = u + 0.02 * np.abs(u).max() * rng.uniform(-1, 1, u.size)
    v, w, du = rng.standard_normal((3, u.size))
    ctx = capi.Context(mesh, p, free, capi.PCEXP_FP64, m_max=2)
    g = ctx.jvp_state_adjoint(u, v, w)
    h = 1e-30
    dJv = (dg.jvp_complex(u + 1j * h * du, v).imag / h) if hasattr(dg, "jvp_complex") else None
    if dJv is None:  # forward-mode J v at complex states through the dual numbers of the oracle
        from oracle import adscalar as ad
        ud = ad.Dual((u + 1j * h * du).reshape(dg.E, dg.nv, dg.N), v.reshape(dg.E, dg.nv, dg.N).astype(complex))
        dJv = (dg.residual(ud).der.imag / h).reshape(-1)
    assert abs(g @ du - w @ dJv) <= 1e-10 * np.linalg.norm(g) * np.linalg.norm(du)
    ctx.close()
