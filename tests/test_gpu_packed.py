"""Contracted 2D kernels on widths around the edges of their packed pairs, V-cell groups and tile
columns (240 compute cells with 8 cells per thread, 112 to 120 with 4), where the source map's
pair order, its padded groups and the clamp fix-ups can go wrong; float32 and 16-bit storage.
Bars: max relative error <= 1e-5 against the float32 oracle (the contracted kernels' bar);
16-bit storage: relative L2 <= 1e-2 (the storage bar)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import TOL, eng, gpu_run, max_rel  # noqa: F401  (eng: fixture)

pytestmark = pytest.mark.gpu

WIDTHS = [3, 4, 5, 7, 8, 9, 12, 111, 112, 113, 119, 121, 239, 240, 241, 247, 249, 480, 485]


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("T,vec,rows", [(1, 8, 2), (4, 8, 2), (6, 8, 2), (8, 8, 1), (8, 8, 2), (8, 4, 2),
                                        (12, 4, 1)])
def test_widths(eng, orc, kind, T, vec, rows):  # noqa: F811
    for n, nx in enumerate(WIDTHS):
        w = synth.make(kind, 2, nx, 21 + n % 3, seed=8100 + 7 * n + kind)
        steps = 2 * T + 1 + n % 2
        g, info = gpu_run(eng, w, steps, T=T, vec=vec, rows=rows, resident=-1)
        assert (info["T"], info["vec"], info["partial_rows"]) == (T, vec, rows)
        o = orc.run(kind, w.u0, w.coef, steps, w.power)
        assert max_rel(g, o) <= TOL, (nx, steps, max_rel(g, o))


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("kind", [0, 1])
def test_widths_16bit(eng, orc, kind, storage):  # noqa: F811
    import torch
    for n, nx in enumerate(WIDTHS):
        w = synth.make(kind, 2, nx, 21, seed=8300 + 7 * n + kind)
        u = torch.from_numpy(w.u0).cuda()
        p = None if w.power is None else torch.from_numpy(w.power).cuda()
        plan = eng.Plan(kind, 2, nx, 21, storage=storage)
        g = plan.run(u, torch.full_like(u, float("nan")), w.coef, 19, power=p).cpu().numpy()
        plan.close()
        o = orc.run(kind, w.u0, w.coef, 19, w.power, dtype=np.float64)
        assert np.linalg.norm(g - o) <= 1e-2 * np.linalg.norm(o), nx


# 3D segments (which planes of which tile columns a block streams): fewer columns than blocks with
# long and short z, about as many, more columns than blocks, one plane, one column; odd widths
# run between padded scratch grids
SHAPES_SEG = [(60, 50, 301), (131, 127, 61), (187, 141, 33), (400, 300, 9), (733, 700, 5), (300, 200, 1),
              (9, 7, 130), (1300, 61, 11)]


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("T,by", [(3, 64), (2, 32)])
def test_segments_3d(eng, orc, kind, T, by):  # noqa: F811
    for n, (nx, ny, nz) in enumerate(SHAPES_SEG):
        w = synth.make(kind, 3, nx, ny, nz, seed=8500 + 7 * n + kind)
        steps = T if n % 2 else 2 * T + 1
        g, info = gpu_run(eng, w, steps, T=T, vec=8, bx=64, by=by)
        assert (info["T"], info["by"]) == (T, by)
        o = orc.run(kind, w.u0, w.coef, steps, w.power)
        assert max_rel(g, o) <= TOL, (nx, ny, nz, steps, max_rel(g, o))


@pytest.mark.parametrize("T", [1, 2, 4])
def test_star_rows(eng, orc, T):  # noqa: F811
    """The streamed radius-2 star: the clamp reaches two cells, so a width may end on a lane's last
    cell or on one of the next lane's first two; heights around the fill of a segment."""
    import torch
    for n, nx in enumerate([1, 2, 7, 8, 9, 10, 239, 240, 241, 242, 247, 248, 249, 490]):
        for ny in (1, 2, 3, 19 + n % 5, 70):
            w = synth.make_star(2, 2, nx, ny, seed=8700 + 7 * n + ny)
            u = torch.from_numpy(w.u0).cuda()
            plan = eng.Plan(0, 2, nx, ny, rad=2, force_T=T)
            steps = 2 * T + 1 + n % 2
            g = plan.run(u, torch.full_like(u, float("nan")), w.coef, steps).cpu().numpy()
            plan.close()
            assert max_rel(g, orc.run_star(2, w.u0, w.coef, steps)) <= TOL, (nx, ny, steps)


@pytest.mark.parametrize("kind,ndim,T,vec,rest", [(0, 2, 8, 8, 1), (0, 2, 8, 8, 3), (1, 2, 8, 8, 2), (1, 2, 8, 4, 1),
                                                  (0, 2, 12, 4, 5), (0, 3, 3, 0, 1), (1, 3, 3, 0, 2), (1, 3, 4, 0, 1),
                                                  (2, 2, 4, 0, 1), (2, 2, 4, 0, 3)])
def test_first_run_captured(eng, orc, kind, ndim, T, vec, rest):  # noqa: F811
    """A plan's first run under stream capture, its last pass shorter than T: nothing may be
    allocated there, so the plan's own kernel runs the few steps.  Replayed, then run plainly."""
    import torch
    nx, ny, nz = (485, 61, 1) if ndim == 2 else (131, 67, 35)
    w = synth.make_vdiff(nx, ny, seed=8900 + T + rest) if kind == 2 else \
        synth.make(kind, ndim, nx, ny, nz, seed=8900 + 7 * T + rest)
    steps = 2 * T + rest
    u = torch.from_numpy(w.u0).cuda()
    p = w.coef if kind == 2 else w.power
    p = None if p is None else torch.from_numpy(p).cuda()
    coef = None if kind == 2 else w.coef
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    out = torch.full_like(u, float("nan"))
    with torch.cuda.stream(s):
        plan = eng.Plan(kind, ndim, nx, ny, nz, force_T=T, force_vec=vec, resident=-1)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            plan.run(u, out, coef, steps, power=p)
        graph.replay()
        s.synchronize()
        g = out.cpu().numpy()
        out.fill_(float("nan"))
        plan.run(u, out, coef, steps, power=p)
        plan.sync()
    assert plan.info()["T"] == T
    plan.close()
    o = orc.run_vdiff2d(w.u0, w.coef, steps) if kind == 2 else orc.run(kind, w.u0, w.coef, steps, w.power)
    assert max_rel(g, o) <= TOL
    assert max_rel(out.cpu().numpy(), o) <= TOL


@pytest.mark.parametrize("kind,ndim", [(0, 2), (1, 2), (0, 3), (1, 3), (2, 2)])
def test_one_scratch_grid(eng, orc, kind, ndim):  # noqa: F811
    """Odd widths without memory for the second scratch grid: the plan is created all the same and
    runs on one (the allocation that fails is injected on the host)."""
    import torch
    nx, ny, nz = (485, 61, 1) if ndim == 2 else (131, 67, 35)
    w = synth.make_vdiff(nx, ny, seed=9100) if kind == 2 else synth.make(kind, ndim, nx, ny, nz, seed=9100 + kind)
    u = torch.from_numpy(w.u0).cuda()
    p = w.coef if kind == 2 else w.power
    p = None if p is None else torch.from_numpy(p).cuda()
    whole = eng.Plan(kind, ndim, nx, ny, nz, resident=-1)
    two = whole.info()["scratch_bytes"]
    whole.close()
    ran = 0
    for n in range(1, 12):
        assert eng.lib.stencil_debug_fail_alloc(n) == eng.ST_OK
        try:
            plan = eng.Plan(kind, ndim, nx, ny, nz, resident=-1)
        except eng.StencilError as e:
            assert e.code == eng.ST_ERR_OOM
            continue
        finally:
            eng.lib.stencil_debug_fail_alloc(0)
        if plan.info()["scratch_bytes"] * 2 == two:
            for steps in (9, 16):
                out = plan.run(u, torch.full_like(u, float("nan")), None if kind == 2 else w.coef, steps, power=p)
                plan.sync()
                o = orc.run_vdiff2d(w.u0, w.coef, steps) if kind == 2 else \
                    orc.run(kind, w.u0, w.coef, steps, w.power)
                assert max_rel(out.cpu().numpy(), o) <= TOL, steps
            ran += 1
        plan.close()
    assert ran >= 1


@pytest.mark.parametrize("rows", [0, 16, 40])
def test_batch_one_pass_in_place(eng, orc, rows):  # noqa: F811
    """Grids of a batch run in place by a single pass (at most 8 steps), cut into several tiles."""
    import torch
    items, refs = [], []
    for i, (nx, ny, steps) in enumerate([(2048, 31, 4), (700, 500, 8), (301, 900, 1), (113, 17, 5), (1, 50, 3)]):
        w = synth.make(i % 2, 2, nx, ny, steps=steps, seed=9200 + i)
        u = torch.from_numpy(w.u0).cuda()
        items.append({"kind": w.kind, "nx": nx, "ny": ny, "steps": steps, "grid_in": u, "grid_out": u,
                      "power": None if w.power is None else torch.from_numpy(w.power).cuda(), "coeffs": w.coef})
        refs.append(orc.run(w.kind, w.u0, w.coef, steps, w.power))
    b = eng.Batch(items, rows_per_item=rows)
    b.run()
    b.sync()
    b.close()
    for it, o in zip(items, refs):
        assert max_rel(it["grid_out"].cpu().numpy(), o) <= TOL, (it["nx"], it["ny"], it["steps"])


@pytest.mark.parametrize("count,lo,hi", [(1, 30, 60), (3, 100, 300), (9, 20, 500), (5, 900, 1500)])
def test_batch_rows(eng, orc, count, lo, hi):  # noqa: F811
    """Batches of few grids take short queue items (16 rows up); heights around an item's."""
    import torch
    rng = np.random.default_rng(count)
    items, refs = [], []
    for i in range(count):
        nx, ny = int(rng.integers(lo, hi)), int(rng.integers(lo, hi))
        if i % 3 == 2:
            ny = ny // 16 * 16 + i % 2
        w = synth.make(i % 2, 2, nx, ny, steps=int(rng.integers(1, 40)), seed=9300 + i)
        u = torch.from_numpy(w.u0).cuda()
        items.append({"kind": w.kind, "nx": nx, "ny": ny, "steps": w.steps, "grid_in": u,
                      "grid_out": torch.full_like(u, float("nan")),
                      "power": None if w.power is None else torch.from_numpy(w.power).cuda(), "coeffs": w.coef})
        refs.append(orc.run(w.kind, w.u0, w.coef, w.steps, w.power))
    b = eng.Batch(items)
    b.run()
    b.sync()
    b.close()
    for it, o in zip(items, refs):
        assert max_rel(it["grid_out"].cpu().numpy(), o) <= TOL, (it["nx"], it["ny"], it["steps"])
