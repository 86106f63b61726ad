"""An exchange of the one-launch Gram-Schmidt columns whose polls run out (limit 0: every wait gives up
at once and returns) ends the call with PCEXP_ERR_TIMEOUT, and the next call gives the same result
as if it had not happened."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    from paper_1801_06300_gb300 import capi as c
    c.load()
    return c


def lost(capi, call):
    with pytest.raises(capi.PcexpError) as e:
        call()
    assert e.value.code == capi.PCEXP_ERR_TIMEOUT
    assert "did not meet in time" in str(e.value)


@pytest.mark.parametrize("form", ["FP64", "FP32_MIXED"])
def test_lost_exchange_is_reported(capi, form):
    case = W.case_vortex2d_small(8)
    ctx = capi.Context(case.mesh, case.p, case.free, getattr(capi, f"PCEXP_{form}"), m_max=case.m)
    ctx.project_state(capi.PCEXP_PROJ_VORTEX, [case.vortex.eps, *case.vortex.center, 10.0])
    u = ctx.get_state()
    b = W.random_coeffs(4, u.shape)

    def step(info):
        return ctx.step(capi.PCEXP_SCHEME_PCEXP, capi.PCEXP_DT_GIVEN, 0.05, case.m, info=info)

    for _ in range(4):  # recorded and replayed steps
        step(False)
    ctx.set_state(u)
    step(True)
    want = ctx.get_state()
    H = ctx.arnoldi(u, b, case.m, want_V=False)[1]

    def good():
        ctx.set_exchange_polls(1 << 23)
        for _ in range(4):
            ctx.set_state(u)
            step(False)
            assert np.array_equal(ctx.get_state(), want)
        assert np.array_equal(ctx.arnoldi(u, b, case.m, want_V=False)[1], H)

    for call in (lambda: ctx.arnoldi(u, b, case.m, want_V=False), lambda: step(True),
                 lambda: (step(False), ctx.get_state()), lambda: (step(False), ctx.synchronize()),
                 lambda: (step(False), ctx.output(0)), lambda: (step(False), ctx.output(1)),
                 lambda: (step(False), step(True)), lambda: [(step(False), ctx.set_state(u)) for _ in range(2)],
                 lambda: ctx.march_steady(capi.PCEXP_SCHEME_EXP1, 10.0, 5.0, 1, case.m)):
        ctx.set_state(u)
        ctx.set_exchange_polls(0)
        lost(capi, call)
        good()
    if form == "FP64":
        ctx.set_exchange_polls(0)
        lost(capi, lambda: ctx.step_backward(u, 0.05, case.m, b))
        good()
    ctx.close()


def test_a_lost_stage_adds_nothing(capi):
    case = W.case_vortex2d_small(8)
    ctx = capi.Context(case.mesh, case.p, case.free, capi.PCEXP_FP64, m_max=case.m)
    ctx.project_state(capi.PCEXP_PROJ_VORTEX, [case.vortex.eps, *case.vortex.center, 10.0])
    u = ctx.get_state()
    ctx.set_exchange_polls(0)
    lost(capi, lambda: ctx.step(capi.PCEXP_SCHEME_EXP1, capi.PCEXP_DT_GIVEN, 0.05, case.m))
    assert np.array_equal(ctx.get_state(), u)
    ctx.close()
