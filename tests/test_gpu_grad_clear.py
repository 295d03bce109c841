"""The backward's accumulators are clear after every call: calls of other sizes and modes, a captured
call launched late and the calls around it give what a new plan gives.  (An 8 x 8 image is one
item, a record's gradient one addition: equal to the bit.)"""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu
CAM = dict(W=8, H=8, fx=9.0, fy=8.5, cx=4.0, cy=4.0, viewmat=np.eye(4))


def _inputs(n):
    g = torch.Generator().manual_seed(100 + n)
    u = lambda lo, hi, *s: (lo + (hi - lo) * torch.rand(s, generator=g)).cuda()
    m3 = torch.stack([u(-0.9, 0.9, n), u(-0.9, 0.9, n), u(0.3, 4, n)], 1)
    pre = raster.preprocess(raster.Plan(), m3, u(-3, -1, n, 3), u(-1, 1, n, 4), u(0.05, 0.6, n), CAM)
    a = (pre["means2D"], pre["conic_opacity"], u(0, 1, n, 3), pre["depths"])
    pl, rg, K = raster.bin_and_sort(raster.Plan(), pre["means2D"], pre["radii"], pre["depths"], 8, 8)
    o = raster.render_forward(raster.Plan(), *a, pl, K, rg, 8, 8, mode="pixel")
    return (*a, pl, K, rg, 8, 8, o["final_T"], o["n_contrib"], u(-1, 1, 3, 8, 8))


def _same(a, b):
    return all(torch.equal(a[k], b[k]) for k in b)


@pytest.mark.parametrize("reserved", [False, True])
def test_calls_of_other_sizes_and_captures(reserved):
    ins = {n: _inputs(n) for n in (1, 40, 3000, 5000)}
    want = {n: raster.render_backward(raster.Plan(), *i, mode="pixel") for n, i in ins.items()}
    assert want[3000]["opacity"].abs().max() > 0
    plan = raster.Plan()
    if reserved:
        plan.reserve(3000, 1 << 16, 64, 64)
    for n in (40, 3000, 1, 3000, 5000, 40, 5000):
        assert _same(raster.render_backward(plan, *ins[n], mode="pixel"), want[n])
    raster.render_backward(plan, *ins[40], mode="static")
    out = {k: torch.empty_like(v) for k, v in want[3000].items()}
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        raster.graph_begin(plan)
        raster.render_backward(plan, *ins[3000], mode="pixel", out=out)
        raster.graph_end(plan)
        assert _same(raster.render_backward(plan, *ins[5000], mode="pixel"), want[5000])
        for n in (40, 5000):
            raster.graph_launch(plan)
            assert _same(raster.render_backward(plan, *ins[n], mode="pixel"), want[n])
            assert _same(out, want[3000])
        raster.graph_launch(plan)
        raster.graph_launch(plan)
    torch.cuda.synchronize()
    assert _same(out, want[3000])
    plan.check()
