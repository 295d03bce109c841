"""Gaussian-wise items by blocks of pixels against pixel-group items: a frame with many segments
takes the first, a crop of the same frame (the same Gaussians, shifted by whole tiles) the
second, and both take the same stops."""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu

N, BIG, CROP, OFF = 1400, (333, 319), (45, 38), (96, 128)


def _render(plan, g, off, size):
    W, H = size
    m, co, col, z = g
    m = m - torch.tensor(off, dtype=torch.float32, device=m.device)  # exact: means are multiples of 1/64
    tiles = -(-W // 16) * -(-H // 16)
    lists = torch.arange(N, dtype=torch.int32).repeat(tiles).cuda()
    first = torch.arange(tiles, dtype=torch.int32) * N
    ranges = torch.stack([first, first + N], 1).contiguous().cuda()
    plan.reset_stats()
    out = raster.render_forward(plan, m.contiguous(), co, col, z, lists, lists.numel(), ranges, W, H, mode="gaussian",
                                n_eval=True)
    plan.check()
    return out, plan.stats()["last_num_items"]


@pytest.mark.parametrize("seg", [256, 512, 2048])
@pytest.mark.parametrize("P", [1, 2, 4, 8, 16])
def test_blocks_and_groups_take_the_same_stops(P, seg):
    rng = np.random.default_rng(11)
    m = np.round(np.stack([rng.uniform(-30, BIG[0] + 30, N), rng.uniform(-30, BIG[1] + 30, N)], 1) * 64) / 64
    s = np.exp(rng.uniform(1.0, 4.7, (N, 2)))
    t = rng.uniform(0, np.pi, N)
    c, n, i0, i1 = np.cos(t), np.sin(t), 1 / s[:, 0] ** 2, 1 / s[:, 1] ** 2
    conic = np.stack([c * c * i0 + n * n * i1, c * n * (i0 - i1), n * n * i0 + c * c * i1], 1)
    o = rng.choice([0.01, 0.05, 0.3, 1.0], N, p=[0.2, 0.3, 0.4, 0.1])
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    g = [f(m), f(np.concatenate([conic, o[:, None]], 1)), f(rng.uniform(0, 1, (N, 3))), f(rng.uniform(1, 5, N))]
    plan = raster.Plan(heavy_threshold=0, gw_pixels=P, gw_segment=seg)
    big, n_big = _render(plan, g, (0, 0), BIG)
    crop, n_crop = _render(plan, g, OFF, CROP)
    segments = -(-N // seg)
    assert n_big == 21 * 20 * segments * 4 and n_crop == 3 * 3 * segments * (256 // P)
    x0, y0 = OFF
    part = {k: v[..., y0:y0 + CROP[1], x0:x0 + CROP[0]] for k, v in big.items()}
    stopped = (crop["n_eval"] < N).float().mean().item()
    assert 0.2 < stopped < 1.0  # (in the first segment where that is the whole list, else in later ones)
    assert torch.equal(part["n_contrib"], crop["n_contrib"]) and torch.equal(part["n_eval"], crop["n_eval"])
    # two float32 products of at most N factors
    assert ((part["final_T"] - crop["final_T"]).abs() <= 3 * N * 2.0 ** -24 * crop["final_T"]).all()
    assert (part["color"] - crop["color"]).abs().max() <= 4 * N * 2.0 ** -24
    assert (part["depth"] - crop["depth"]).abs().max() <= 5 * 4 * N * 2.0 ** -24
