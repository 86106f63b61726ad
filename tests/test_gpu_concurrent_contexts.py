"""Contexts stepped at the same time by a thread each, on streams of their own, give the results they give
alone: the grids of their one-launch Gram-Schmidt columns meet on the SMs."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["FP64", "FP32_MIXED"])
def test_threads_and_streams(form):
    import torch
    from paper_1801_06300_gb300 import capi
    capi.load()
    sizes = [(4, 1), (16, 1), (24, 2), (48, 2), (16, 1), (96, 2)]  # elements per side, p
    streams = [torch.cuda.Stream() for _ in sizes]
    ctxs, starts = [], []
    for (n, p), st in zip(sizes, streams):
        c = capi.Context(W.periodic_square(n, 10.0, 0.1, 3), p, W.Freestream(0.45, 20.0), getattr(capi, f"PCEXP_{form}"),
                         m_max=20, stream=st.cuda_stream)
        c.project_state(capi.PCEXP_PROJ_VORTEX, [5.0, 5.0, 5.0, 10.0])
        ctxs.append(c)
        starts.append(c.get_state())

    def run(i, out):
        ctxs[i].set_state(starts[i])
        for _ in range(6):
            ctxs[i].step(capi.PCEXP_SCHEME_PCEXP, capi.PCEXP_DT_GLOBAL_CFL, 1.0, 20, info=False)
        out[i] = ctxs[i].get_state()

    alone, together = [None] * len(sizes), [None] * len(sizes)
    for i in range(len(sizes)):
        run(i, alone)
    for _ in range(3):
        threads = [threading.Thread(target=run, args=(i, together)) for i in range(len(sizes))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for a, b in zip(alone, together):
            assert b is not None and np.array_equal(a, b)
    for c in ctxs:
        c.close()
