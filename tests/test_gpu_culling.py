"""The records that the persistent kernels skip for a block of pixels contribute to none of its
pixels: against the static kernels, which visit every record, the transmittances and
contributor counts are the same bits, for thin, large, faint and off-screen Gaussians and
conics that are not positive definite."""
import math

import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu

W, H, TILE, N = 70, 45, (16, 16), 1500


def _gaussians(kind, seed=0):
    rng = np.random.default_rng([seed, ["thin", "mixed", "faint", "degenerate"].index(kind)])
    m = np.stack([rng.uniform(-60, W + 60, N), rng.uniform(-60, H + 60, N)], 1)
    lo, hi = (0.55, 400.0) if kind == "thin" else (0.55, 40.0)
    s = np.exp(rng.uniform(math.log(lo), math.log(hi), (N, 2)))
    if kind == "thin":
        s[:, 1] = 0.55
    t = rng.uniform(0, math.pi, N)
    c, n = np.cos(t), np.sin(t)
    i0, i1 = 1 / s[:, 0] ** 2, 1 / s[:, 1] ** 2
    conic = np.stack([c * c * i0 + n * n * i1, c * n * (i0 - i1), n * n * i0 + c * c * i1], 1)
    o = rng.uniform(0.004, 0.3, N)
    if kind == "faint":  # around the 1/255 threshold
        o = (1 + rng.choice([-1e-3, 1e-6, 1e-3, 0.1], N)) / 255
    if kind == "degenerate":  # det <= 0 (a ridge or a saddle) for every third Gaussian
        conic[::3, 1] = np.sqrt(conic[::3, 0] * conic[::3, 2]) * rng.uniform(1.0, 1.02, conic[::3].shape[0])
    g = [m, np.concatenate([conic, o[:, None]], 1), rng.uniform(0, 1, (N, 3)), rng.uniform(1, 5, N)]
    return [torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda() for a in g]


@pytest.mark.parametrize("rows", [1, 2, 4, 8])
@pytest.mark.parametrize("kind", ["thin", "mixed", "faint", "degenerate"])
def test_skipped_records_contribute_nothing(kind, rows):
    m, co, col, z = _gaussians(kind)
    tiles = -(-W // 16) * -(-H // 16)
    lists = torch.arange(N, dtype=torch.int32).repeat(tiles).cuda()
    first = torch.arange(tiles, dtype=torch.int32) * N
    ranges = torch.stack([first, first + N], 1).contiguous().cuda()
    plan = raster.Plan(pixel_rows=rows, heavy_threshold=2147483647)
    grad = torch.from_numpy(np.random.default_rng(1).normal(0, 1, (3, H, W)).astype(np.float32)).cuda()
    out, grads = {}, {}
    for mode in ("static", "pixel"):
        out[mode] = raster.render_forward(plan, m, co, col, z, lists, lists.numel(), ranges, W, H, mode=mode, n_eval=True)
        grads[mode] = raster.render_backward(plan, m, co, col, z, lists, lists.numel(), ranges, W, H,
                                             out[mode]["final_T"], out[mode]["n_contrib"], grad, mode=mode)
    plan.check()
    a, b = out["static"], out["pixel"]
    for k in ("final_T", "n_contrib", "n_eval"):
        assert torch.equal(a[k], b[k]), k
    # the same terms in the same order: N roundings of a sum of at most 1 (colour) or 5 (depth)
    assert (a["color"] - b["color"]).abs().max() <= N * 2.0 ** -24
    assert (a["depth"] - b["depth"]).abs().max() <= 5 * N * 2.0 ** -24
    for k in ("means2D", "conic", "opacity", "colors"):  # the same terms in another order
        x, y = grads["static"][k].double(), grads["pixel"][k].double()
        assert (x - y).norm() <= 1e-4 * x.norm(), k
