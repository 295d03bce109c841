"""Two records at a time (pixel-wise items, windows without an odd record) against the static
kernel, which takes one: windows of odd and even counts, stops at the first and at the second of
a pair, several of a lane's pixels at different records, windows with an odd record."""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu
W, H = 35, 50


@pytest.mark.parametrize("odd", [None, 0, -1])
@pytest.mark.parametrize("rows", [1, 2, 4, 8])
@pytest.mark.parametrize("n", [1, 2, 3, 32, 33, 70])
def test_two_records_stop_as_one(n, rows, odd):
    rng = np.random.default_rng([n, rows])
    s = rng.uniform(4, 30, n)
    o = rng.uniform(0.2, 0.985, n)
    if odd is not None:
        o[odd] = 1.0  # the clamp decides
    m = np.stack([rng.uniform(0, W, n), rng.uniform(0, H, n)], 1)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    g = (f(m), f(np.stack([1 / s ** 2, 0 * s, 1 / s ** 2, o], 1)), f(rng.uniform(0, 1, (n, 3))), f(rng.uniform(1, 5, n)))
    tiles = -(-W // 16) * -(-H // 16)
    lists = torch.arange(n, dtype=torch.int32).repeat(tiles).cuda()
    first = torch.arange(tiles, dtype=torch.int32) * n
    ranges = torch.stack([first, first + n], 1).contiguous().cuda()
    out = {}
    for mode in ("pixel", "static"):
        plan = raster.Plan(pixel_rows=rows)
        out[mode] = raster.render_forward(plan, *g, lists, lists.numel(), ranges, W, H, mode=mode, n_eval=True)
        plan.check()
    a, b = out["pixel"], out["static"]
    assert n < 32 or 0.2 < (b["n_eval"] < n).float().mean() <= 1.0
    assert all(torch.equal(a[k], b[k]) for k in ("n_contrib", "n_eval", "final_T", "alpha"))
    # the same products added in the same order, at most with another contraction: n terms below 1 and 5
    assert (a["color"] - b["color"]).abs().max() <= 4 * n * 2.0 ** -24
    assert (a["depth"] - b["depth"]).abs().max() <= 5 * 4 * n * 2.0 ** -24
