"""The library's tables and flags reach the device in the order of the stream that reads them.

A pageable host-to-device copy (or a memset) on the null stream may return before it has landed,
and a non-blocking stream does not wait for the null stream, so a kernel launched next could read
what the buffer held before: for a list of segments, out-of-range addresses."""
import glob
import os
import re

import numpy as np
import pytest

import synth
from test_gpu_parity import TOL, eng, max_rel  # noqa: F401  (eng: fixture)

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_00438_gb300", "csrc")


def test_no_upload_on_the_null_stream():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(f).read(), flags=re.S)
        assert not re.search(r"\bcudaMemset\s*\(", src), f
        for call in re.findall(r"\bcudaMemcpy\s*\([^;]*;", src):
            assert "cudaMemcpyDeviceToHost" in call, (f, call)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,ndim,rad", [(0, 2, 1), (1, 2, 1), (0, 3, 1), (1, 3, 1), (2, 2, 1), (0, 2, 2)])
def test_first_run_on_a_side_stream(eng, orc, kind, ndim, rad):  # noqa: F811
    """First calls of plans on a non-blocking stream while the null stream has work queued: the
    plan's own kernel, then one whose last pass is shorter."""
    import torch
    nx, ny, nz = (485, 333, 1) if ndim == 2 else (131, 67, 35)
    w = synth.make_star(2, 2, nx, ny, seed=9400) if rad == 2 else \
        synth.make_vdiff(nx, ny, seed=9400) if kind == 2 else synth.make(kind, ndim, nx, ny, nz, seed=9400 + kind)
    u = torch.from_numpy(w.u0).cuda()
    p = w.coef if kind == 2 else w.power if rad < 2 else None
    p = None if p is None else torch.from_numpy(p).cuda()
    coef = None if kind == 2 else w.coef
    s = torch.cuda.Stream()
    busy = torch.empty(1 << 28, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        out = torch.full_like(u, float("nan"))
    for _ in range(8):
        busy.add_(1.0)
    with torch.cuda.stream(s):
        plan = eng.Plan(kind, ndim, nx, ny, nz, rad=rad if rad > 1 else 0, resident=-1)
        for steps in (plan.info()["T"], 2 * plan.info()["T"] + 1):
            plan.run(u, out, coef, steps, power=p)
            plan.sync()
            o = orc.run_star(2, w.u0, w.coef, steps) if rad == 2 else \
                orc.run_vdiff2d(w.u0, w.coef, steps) if kind == 2 else orc.run(kind, w.u0, w.coef, steps, w.power)
            assert max_rel(out.cpu().numpy(), o) <= TOL, steps
        plan.close()
