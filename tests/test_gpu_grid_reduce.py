"""The last-block reductions of the density norm, the time step and the entropy error against the
oracle for one block, a few, and more elements than the largest grid has threads (608 blocks)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,p", [("channel", 1, 0), ("square", 16, 0), ("square", 17, 1), ("square", 160, 0),
                                      ("square", 280, 0), ("cube", 3, 2)])
def test_reductions_match_oracle(kind, n, p):
    from oracle.dg import DGOracle
    from paper_1801_06300_gb300 import capi
    mesh = (W.bump_channel(1, 1, 0.0, 1) if kind == "channel" else W.periodic_square(n, 10.0, 0.1, 3) if kind == "square"
            else W.periodic_cube_kuhn(n, 10.0, 0.1, 5))
    capi.load()
    free = W.Freestream(mach=0.45, alpha_deg=12.0)
    dg = DGOracle(mesh, p, free)
    u = dg.project(lambda x: np.broadcast_to(dg.freestream_state(), x.shape[:-1] + (dg.nv,)))
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(3, u.shape)).reshape(-1)
    volume = float(np.sum(dg.area))
    r = dg.state_at(dg.residual(u), dg.rq, local=True)[..., 0]
    res = np.sqrt(np.sum(dg.wq * r ** 2)) / volume
    ctx = capi.Context(mesh, p, free, capi.PCEXP_FP64, m_max=2)
    for _ in range(2):  # the counters are left ready for the next call
        ctx.set_state(u)
        info = ctx.step(capi.PCEXP_SCHEME_EXP1, capi.PCEXP_DT_GLOBAL_CFL, 0.5, 2)
        # up to 156,800 terms of one sign: the sum's rounding is below 1e-12, R's relative error (a
        # perturbation of 2% in each coefficient) too
        assert abs(info["res_norm"] - res) <= 1e-11 * res
        dt = float(np.min(dg.local_dt(u, 0.5)))
        assert abs(info["dt"] - dt) <= 1e-13 * dt
    ctx.set_state(u)
    want = dg.entropy_error(u, volume)
    got = ctx.output(1)
    assert abs(got - want) <= 1e-9 * want  # sqrt(sum / volume - 1): cancels about four digits
    ctx.close()
