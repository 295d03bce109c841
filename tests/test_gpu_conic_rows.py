"""Gradients of conic_opacity as one array of rows against the separate arrays: written by the
render backward (an 8 x 8 image is one item: a record's gradient is one addition, so
equal to the bit) and read by the projection backward, also from a view that is strided or starts
off a 16-byte boundary."""
import numpy as np
import pytest
import torch

from paper_2412_17378_gb300 import raster

pytestmark = pytest.mark.gpu
CAM = dict(W=8, H=8, fx=9.0, fy=8.5, cx=4.0, cy=4.0, viewmat=np.eye(4))


def _scene(n):
    g = torch.Generator().manual_seed(n)
    u = lambda lo, hi, *s: (lo + (hi - lo) * torch.rand(s, generator=g)).cuda()
    m3 = torch.stack([u(-0.9, 0.9, n), u(-0.9, 0.9, n), u(-0.3, 4, n)], 1)  # (some are culled)
    return m3, u(-3, -1, n, 3), u(-1, 1, n, 4), u(0.05, 0.9, n), u(0, 1, n, 3), u(-1, 1, 3, 8, 8)


def _backward(plan, s, mode, out=None):
    m3, ls, q, op, col, up = s
    pre = raster.preprocess(plan, m3, ls, q, op, CAM)
    a = (pre["means2D"], pre["conic_opacity"], col, pre["depths"])
    pl, rg, K = raster.bin_and_sort(plan, pre["means2D"], pre["radii"], pre["depths"], 8, 8)
    o = raster.render_forward(plan, *a, pl, K, rg, 8, 8, mode=mode)
    g = raster.render_backward(plan, *a, pl, K, rg, 8, 8, o["final_T"], o["n_contrib"], up, mode=mode, out=out)
    return pre["radii"], g


@pytest.mark.parametrize("mode", ["pixel", "gaussian"])
@pytest.mark.parametrize("n", [1, 2, 31, 300])
def test_render_backward_rows(n, mode):
    plan, s = raster.Plan(heavy_threshold=0), _scene(n)
    _, g = _backward(plan, s, mode)
    e = lambda *shape: torch.full(shape, 7.0, device="cuda")
    _, r = _backward(plan, s, mode, dict(means2D=e(n, 2), conic_opacity=e(n, 4), colors=e(n, 3), depths=e(n)))
    assert torch.equal(r["conic_opacity"], torch.cat([g["conic"], g["opacity"][:, None]], 1))
    assert all(torch.equal(r[k], g[k]) for k in ("means2D", "colors", "depths"))
    assert n < 31 or g["opacity"].abs().max() > 0


@pytest.mark.parametrize("view", ["rows", "off", "strided", "expanded", "none"])
@pytest.mark.parametrize("n", [1, 129, 1000])
def test_projection_backward_rows(n, view):
    plan, (m3, ls, q, op, _, _) = raster.Plan(), _scene(n)
    gco = torch.linspace(-2, 3, 4 * n, device="cuda").reshape(n, 4)
    if view == "off":
        buf = torch.zeros(4 * n + 1, device="cuda")
        buf[1:] = gco.reshape(-1)
        gco = buf[1:].reshape(n, 4)
    if view == "strided":
        gco = gco.t().contiguous().t()
    if view == "expanded":
        gco = torch.tensor(0.5, device="cuda").expand(n, 4)
    leaves = [t.clone().requires_grad_(True) for t in (m3, ls, q, op)]
    m2, co, z, radii = raster.PreprocessFunction.apply(*leaves, plan, CAM, (16, 16))
    gm, gz = torch.linspace(-1, 1, 2 * n, device="cuda").reshape(n, 2), torch.linspace(0, 1, n, device="cuda")
    if view == "none":
        torch.autograd.backward([m2, z], [gm, gz])
        gco = torch.zeros(n, 4, device="cuda")
    else:
        torch.autograd.backward([m2, co, z], [gm, gco, gz])
    want = raster.preprocess_backward(plan, m3, ls, q, CAM, radii, gm, gco[:, :3].contiguous(), gz)
    got = dict(zip(("means3D", "log_scales", "quats"), (t.grad for t in leaves)))
    assert all(torch.equal(got[k], want[k]) for k in want)
    assert torch.equal(leaves[3].grad, gco[:, 3])
