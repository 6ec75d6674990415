"""The grids a plan of odd width takes besides those it needs (a second padded scratch grid, the
padded power map of 3D Hotspot): they never make a creation fail that would succeed without them,
and they leave most of the free memory alone."""
import pytest

import synth
from test_gpu_parity import TOL, eng, max_rel  # noqa: F401  (eng: fixture)

pytestmark = pytest.mark.gpu

SHAPES = {2: (485, 61, 1), 3: (131, 67, 35)}


@pytest.mark.parametrize("kind,ndim,rad", [(0, 2, 0), (1, 2, 0), (0, 3, 0), (1, 3, 0), (2, 2, 0), (0, 2, 2)])
def test_extra_grids_come_last(eng, kind, ndim, rad):  # noqa: F811
    """Fail each allocation of a creation in turn: those the plan needs come first, and from the
    first that it can do without on, every creation succeeds."""
    created = []
    for n in range(1, 24):
        assert eng.lib.stencil_debug_fail_alloc(n) == eng.ST_OK
        try:
            plan = eng.Plan(kind, ndim, *SHAPES[ndim], rad=rad, resident=-1)
            plan.close()
            created.append(True)
        except eng.StencilError as e:
            assert e.code == eng.ST_ERR_OOM
            created.append(False)
        finally:
            eng.lib.stencil_debug_fail_alloc(0)
    need = created.index(True)
    assert need >= 2 and all(created[need:]), created


def test_little_free_memory(eng, orc):  # noqa: F811
    """With 2 GiB of device memory free, a plan whose extra grids would take 0.5 GiB runs on one."""
    import torch
    nx, ny, nz = 513, 512, 256
    torch.cuda.empty_cache()
    plan = eng.Plan(1, 3, nx, ny, nz)
    two = plan.info()["scratch_bytes"]
    plan.close()
    w = synth.make(1, 3, nx, ny, 6, seed=9500)
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    try:
        plan = eng.Plan(1, 3, nx, ny, nz)
        assert plan.info()["scratch_bytes"] * 2 == two
        plan.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    u, p = torch.from_numpy(w.u0).cuda(), torch.from_numpy(w.power).cuda()
    plan = eng.Plan(1, 3, nx, ny, 6)
    out = plan.run(u, torch.full_like(u, float("nan")), w.coef, 7, power=p)
    plan.sync()
    assert max_rel(out.cpu().numpy(), orc.run(1, w.u0, w.coef, 7, w.power)) <= TOL
    plan.close()


@pytest.mark.parametrize("kind,ndim,nx,ny,nz,kw,holds", [
    (0, 2, 256, 192, 1, {}, 3),             # resident tiles: exchange grids, counters, flag
    (0, 2, 300, 200, 1, {"exact": True}, 3),
    (1, 2, 1024, 1024, 1, {"resident": 1}, 4),   # (and the source map)
    (0, 2, 484, 61, 1, {"resident": -1}, 3),     # passes: scratch, one list of segments, flag
    (0, 3, 132, 67, 35, {}, 3), (2, 2, 484, 61, 1, {}, 3), (0, 2, 484, 61, 1, {"rad": 2}, 3)])
def test_creation_prepares_what_runs(eng, kind, ndim, nx, ny, nz, kw, holds):  # noqa: F811
    """No segments for passes that a plan may never run: none for resident tiles, none for remainder
    passes."""
    live = eng.lib.stencil_debug_live_allocs()
    plan = eng.Plan(kind, ndim, nx, ny, nz, **kw)
    assert eng.lib.stencil_debug_live_allocs() - live == holds, plan.info()
    plan.close()
    assert eng.lib.stencil_debug_live_allocs() == live
