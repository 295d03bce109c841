"""Records and pixels that the persistent kernels take through the pair rule in full (alpha
clamp, near-singular conics, colours and gradients that are not finite), mixed with ordinary
ones: decisions are the static kernels' bit for bit, and a value that is not finite reaches
the same outputs."""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu

W, H, N = 44, 37, 900


def _inputs(kind):
    rng = np.random.default_rng([7, ["opaque", "thin", "colour", "gradient"].index(kind)])
    m = np.stack([rng.uniform(-4, W + 4, N), rng.uniform(-4, H + 4, N)], 1)
    s = np.exp(rng.uniform(0.0, 2.0, (N, 2)))
    if kind == "thin":  # det around 1e-5 a c, on both sides
        s[::2] = np.stack([np.full(len(s[::2]), 300.0), rng.uniform(0.3, 2.0, len(s[::2]))], 1)
    t = rng.uniform(0, np.pi, N)
    c, n, i0, i1 = np.cos(t), np.sin(t), 1 / s[:, 0] ** 2, 1 / s[:, 1] ** 2
    conic = np.stack([c * c * i0 + n * n * i1, c * n * (i0 - i1), n * n * i0 + c * c * i1], 1)
    o = rng.uniform(0.01, 0.2, N)
    if kind == "opaque":
        o[::3] = rng.choice([0.98, 0.99, 0.995, 1.0], len(o[::3]))
    col, z = rng.uniform(0, 1, (N, 3)), rng.uniform(1, 5, N)
    if kind == "colour":
        col[::97, 1] = rng.choice([np.nan, np.inf, -np.inf, 1e30], len(col[::97]))
        z[50::101] = np.inf
    grad = rng.normal(0, 1, (3, H, W))
    if kind == "gradient":
        grad[0, 5, 7], grad[2, 30, 40], grad[1, 20, 3] = np.nan, np.inf, 1e30
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    return [f(m), f(np.concatenate([conic, o[:, None]], 1)), f(col), f(z)], f(grad)


@pytest.mark.parametrize("rows", [1, 2, 4, 8])
@pytest.mark.parametrize("kind", ["opaque", "thin", "colour", "gradient"])
def test_odd_records_follow_the_pair_rule(kind, rows):
    g, grad = _inputs(kind)
    tiles = -(-W // 16) * -(-H // 16)
    lists = torch.arange(N, dtype=torch.int32).repeat(tiles).cuda()
    first = torch.arange(tiles, dtype=torch.int32) * N
    ranges = torch.stack([first, first + N], 1).contiguous().cuda()
    plan = raster.Plan(pixel_rows=rows, heavy_threshold=2147483647)
    out, grads = {}, {}
    # the static kernel always carries the depth's terms: with a depth that is not finite the other
    # has to be asked for them too
    more = dict(dL_ddepth=torch.zeros_like(grad[0]), dL_dalpha=torch.zeros_like(grad[0])) if kind == "colour" else {}
    for mode in ("static", "pixel"):
        out[mode] = raster.render_forward(plan, *g, lists, lists.numel(), ranges, W, H, mode=mode, n_eval=True)
        grads[mode] = raster.render_backward(plan, *g, lists, lists.numel(), ranges, W, H, out[mode]["final_T"],
                                             out[mode]["n_contrib"], grad, mode=mode, **more)
    plan.check()
    a, b = out["static"], out["pixel"]
    for k in ("final_T", "n_contrib", "n_eval"):
        assert torch.equal(a[k], b[k]), k
    for x, y in [(a["color"], b["color"]), (a["depth"], b["depth"])] + [
            (grads["static"][k], grads["pixel"][k]) for k in ("means2D", "conic", "opacity", "colors")]:
        fine = torch.isfinite(x)
        assert torch.equal(fine, torch.isfinite(y))
        # finite values: the same terms, in another order for the gradients; 1e30 among them
        # takes its neighbours' share of float32, so element by element against the largest
        big = fine & (x.abs() < 1e20)
        assert torch.equal(big, fine & (y.abs() < 1e20))
        d = (x[big].double() - y[big].double()).norm()
        assert d <= 1e-4 * x[big].double().norm() + 1e-12
