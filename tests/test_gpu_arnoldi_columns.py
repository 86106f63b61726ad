"""FP32 Gram-Schmidt passes for every number of columns up to 31 and vector lengths below, around and
above one wave of tiles: orthonormality and the Arnoldi relation, with the second pass where the first
cancelled and on every column."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "K72": lambda: (W.periodic_square(3, 10.0, 0.1, 3), 0),
    "K600": lambda: (W.periodic_square(5, 10.0, 0.1, 3), 1),
    "K13824": lambda: (W.periodic_square(24, 10.0, 0.1, 3), 1),
    "K414720": lambda: (W.periodic_square(72, 10.0, 0.1, 3), 3),
    "K960000": lambda: (W.periodic_cube_kuhn(20, 10.0, 0.1, 5, periodic=False), 1),
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("reorth", ["SELECTIVE", "ALWAYS"])
def test_fp32_columns(name, reorth):
    from paper_1801_06300_gb300 import capi
    mesh, p = MESHES[name]()
    capi.load()
    m = 31
    ctx = capi.Context(mesh, p, W.Freestream(0.45, 20.0), capi.PCEXP_FP32_MIXED, m_max=m,
                       reorth=getattr(capi, f"PCEXP_REORTH_{reorth}"))
    u = ctx.get_state().reshape(ctx.E, ctx.nv, ctx.nb)
    u = (u + 0.02 * np.abs(u[:, :, :1]) * W.random_coeffs(3, u.shape)).reshape(-1)
    V, H, k, beta = ctx.arnoldi(u, W.random_coeffs(4, u.shape), m)
    assert k == m
    # 1e-5 and 2e-5: the FP32 form's bounds on orthonormality and on the relation (its J v is
    # computed again here, in the same arithmetic)
    assert np.abs(V @ V.T - np.eye(m + 1)).max() <= 1e-5
    for j in range(m):
        jv = ctx.jvp(u, V[j])
        assert np.linalg.norm(H[: j + 2, j] @ V[: j + 2] - jv) <= 2e-5 * np.linalg.norm(jv), j
    ctx.close()
