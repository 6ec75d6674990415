"""A plan's first run under stream capture prepares the kernels that a plain run uses, its remainder
pass among them: a plain run after it allocates nothing more and gives the same bits."""
import numpy as np
import pytest

import synth
from test_gpu_parity import TOL, eng, max_rel  # noqa: F401  (eng: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocking", [False, True])
@pytest.mark.parametrize("kind,ndim,rad,T,vec,rest", [(0, 2, 0, 8, 8, 1), (0, 2, 0, 8, 8, 4), (1, 2, 0, 8, 8, 3),
                                                      (1, 2, 0, 8, 4, 3), (0, 3, 0, 3, 0, 1), (1, 3, 0, 3, 0, 2),
                                                      (2, 2, 0, 4, 0, 2), (0, 2, 2, 4, 0, 2), (0, 2, 2, 4, 0, 1)])
def test_remainder_prepared_under_capture(eng, orc, kind, ndim, rad, T, vec, rest, blocking):  # noqa: F811
    import ctypes
    import torch
    nx, ny, nz = (484, 61, 1) if ndim == 2 else (132, 67, 35)
    w = synth.make_star(2, 2, nx, ny, seed=9600 + rest) if rad == 2 else \
        synth.make_vdiff(nx, ny, seed=9600 + rest) if kind == 2 else \
        synth.make(kind, ndim, nx, ny, nz, seed=9600 + 7 * T + rest)
    steps = 2 * T + rest
    u = torch.from_numpy(w.u0).cuda()
    p = w.coef if kind == 2 else None if rad == 2 else w.power
    p = None if p is None else torch.from_numpy(p).cuda()
    coef = None if kind == 2 else w.coef
    out, again = torch.full_like(u, float("nan")), torch.full_like(u, float("nan"))
    torch.cuda.synchronize()
    raw = None
    if blocking:   # a stream that the null stream waits for
        rt = ctypes.CDLL("libcudart.so")
        raw = ctypes.c_void_p()
        assert rt.cudaStreamCreate(ctypes.byref(raw)) == 0
        s = torch.cuda.ExternalStream(raw.value)
    else:
        s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        plan = eng.Plan(kind, ndim, nx, ny, nz, rad=rad, force_T=T, force_vec=vec, resident=-1)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            plan.run(u, out, coef, steps, power=p)
        live = eng.lib.stencil_debug_live_allocs()
        graph.replay()
        graph.replay()
        s.synchronize()
        g = out.cpu().numpy()
        plan.run(u, again, coef, steps, power=p)
        plan.sync()
    assert eng.lib.stencil_debug_live_allocs() == live
    o = orc.run_star(2, w.u0, w.coef, steps) if rad == 2 else \
        orc.run_vdiff2d(w.u0, w.coef, steps) if kind == 2 else orc.run(kind, w.u0, w.coef, steps, w.power)
    assert max_rel(g, o) <= TOL
    assert np.array_equal(g, again.cpu().numpy())
    del graph
    plan.close()
