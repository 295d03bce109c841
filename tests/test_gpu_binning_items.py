"""The scatter's passes, batches and items: groups hit by most of a block's Gaussians (more than a
batch), by a few, and by none; blocks below, at and above a pass of 2048; tile grids that end
inside a group.  Complete lists are the stable depth order per tile, truncated ones prefixes."""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu


def _scene(kind, n, W, H):
    rng = np.random.default_rng([3, n, ["dense", "sparse", "mixed"].index(kind)])
    m = np.stack([rng.uniform(0, W, n), rng.uniform(0, H, n)], 1).astype(np.float32)
    r = rng.integers(1, 9, n)
    if kind == "dense":
        r[:] = 400
    if kind == "mixed":  # half of them on one corner
        m[::2] = rng.uniform(0, 40, (len(m[::2]), 2))
        r[rng.random(n) < 0.02] = 300
    z = rng.choice(np.linspace(1, 5, 64), n).astype(np.float32)  # many ties
    s = np.maximum(r / 3.0, 0.6)
    conic = np.stack([1 / s ** 2, 0 * s, 1 / s ** 2, rng.uniform(0.3, 0.99, n)], 1).astype(np.float32)
    return m, r.astype(np.int32), z, conic


def _expected(m, r, z, W, H):
    tx, ty = -(-W // 16), -(-H // 16)
    q = lambda a, hi: np.clip(np.floor(a.astype(np.float32) / np.float32(16)), 0, hi).astype(int)
    rf = r.astype(np.float32)
    x0, x1 = q(m[:, 0] - rf, tx), q(m[:, 0] + (rf + np.float32(15)), tx)
    y0, y1 = q(m[:, 1] - rf, ty), q(m[:, 1] + (rf + np.float32(15)), ty)
    order = np.argsort(z, kind="stable")
    lists = []
    for t in range(tx * ty):
        x, y = t % tx, t // tx
        o = order[(x0[order] <= x) & (x < x1[order]) & (y0[order] <= y) & (y < y1[order])]
        lists.append(o)
    return lists


@pytest.mark.parametrize("block", [0, 64, 544, 2048, 4096])
@pytest.mark.parametrize("kind,n,W,H", [("dense", 2600, 150, 90), ("dense", 9000, 64, 48), ("sparse", 9000, 500, 333),
                                        ("mixed", 7001, 301, 77), ("sparse", 1, 33, 17)])
def test_lists_of_all_items(kind, n, W, H, block):
    m, r, z, conic = _scene(kind, n, W, H)
    want = _expected(m, r, z, W, H)
    d = lambda a: torch.from_numpy(a).cuda()
    plan = raster.Plan(bin_block=block)
    buf = torch.zeros(sum(map(len, want)) + 8, dtype=torch.int32, device="cuda")
    pl, rg, K = raster.bin_and_sort(plan, d(m), d(r), d(z), W, H, point_list=buf)
    assert K == sum(map(len, want))
    pl, rg = pl.cpu().numpy(), rg.cpu().numpy()
    for t, w in enumerate(want):
        np.testing.assert_array_equal(pl[rg[t, 0]:rg[t, 1]], w)
    cut, rg, K2 = raster.bin_and_sort(plan, d(m), d(r), d(z), W, H, conic_opacity=d(conic))
    assert K2 <= K
    cut, rg = cut.cpu().numpy(), rg.cpu().numpy()
    for t, w in enumerate(want):
        got = cut[rg[t, 0]:rg[t, 1]]
        np.testing.assert_array_equal(got, w[:len(got)])
        assert len(got) or not len(w)
    plan.check()
