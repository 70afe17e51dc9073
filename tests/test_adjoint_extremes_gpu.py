"""The adjoint at the ends of its input range on the GPU: colour maps with non-finite entries that no
sample reads, gradients that overflow, checkpoints with rays that took no sample.  Each is compared
with a run on ordinary values of the same shape, so only what must be unaffected is asserted."""
import numpy as np
import pytest
import torch

import scene
from parity import shw, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    return shw()


def _backward(m, cube, cam, lut, g, scale, edit=None, **kw):
    out = m.render(cube, cam, "composite", lut=lut, opacity_scale=scale, ckpt=True, **kw)
    if edit is not None:
        edit(out["ckpt"])
    gv, gl, gs = torch.zeros_like(cube), torch.zeros_like(lut), torch.zeros(1, device="cuda")
    m.render_backward(cube, cam, g, out["ckpt"], lut=lut, opacity_scale=scale, grad_vol=gv, grad_lut=gl, grad_scale=gs, **kw)
    m.sync_status()
    return gv, gl, float(gs.item())


@pytest.mark.parametrize("interp", ["trilinear", "nearest"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_knots_that_no_sample_reads(m, interp, value):
    """Voxels in [0.25, 0.75] of the domain [0, 1] read knots 63 to 192: knots 0 and 1 may hold anything."""
    dims = (24, 20, 28)
    cube = 0.25 + 0.5 * torch.rand(dims[::-1], generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    cam = scene.orbit_camera(dims, 30, 20, 50, 41)  # rays of different lengths in every warp
    g = torch.rand((41, 50, 4), generator=torch.Generator("cuda").manual_seed(4), device="cuda")
    lut = to_dev(scene.linear_lut())
    bad = lut.clone()
    bad[:2] = value
    kw = dict(lo=0.0, hi=1.0, interp=interp)
    _, _, want = _backward(m, cube, cam, lut, g, 0.05, **kw)
    gv, gl, gs = _backward(m, cube, cam, bad, g, 0.05, **kw)
    assert bool(torch.isfinite(gv).all()) and bool(torch.isfinite(gl).all())
    assert gs == pytest.approx(want, rel=1e-4)  # (the sums' order varies)


def test_scale_gradient_that_overflows(m):
    """One pixel at the image's centre (the first tile that any warp takes; the image has more tiles than
    the device has warps) whose gradients overflow: the sum is infinite, not NaN."""
    dims = (24, 24, 24)
    cube = 0.25 + 0.5 * torch.rand(dims, generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    cam = scene.orbit_camera(dims, 0, 0, 640, 640)
    lut = to_dev(scene.linear_lut())
    g = torch.zeros((640, 640, 4), device="cuda")
    g[..., 3] = 1.0
    g[320, 320, 3] = 3e38  # times 20 and more samples' alpha
    _, _, gs = _backward(m, cube, cam, lut, g, 0.05, lo=0.0, hi=1.0)
    assert gs == np.inf


def test_checkpoints_without_samples(m):
    """A checkpoint whose count for some pixels is zero or negative: those rays give nothing, and the
    others what they gave."""
    dims = (24, 20, 28)
    cube = 0.25 + 0.5 * torch.rand(dims[::-1], generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    cam = scene.orbit_camera(dims, 30, 20, 50, 41)
    lut = to_dev(scene.linear_lut())
    g = torch.rand((41, 50, 4), generator=torch.Generator("cuda").manual_seed(4), device="cuda")

    def counts(value):
        def edit(ckpt):
            ckpt[:4 * 41 * 50].view(torch.int32)[7::13] = value
        return edit

    zero, negative = (_backward(m, cube, cam, lut, g, 0.05, edit=counts(v), lo=0.0, hi=1.0) for v in (0, -1))
    for a, b in zip(zero[:2], negative[:2]):
        assert float(a.abs().max()) > 0 and torch.allclose(a, b, rtol=1e-4, atol=1e-6 * float(a.abs().max()))
    assert zero[2] != 0.0 and negative[2] == pytest.approx(zero[2], rel=1e-4)


@pytest.mark.parametrize("interp", ["trilinear", "nearest"])
def test_more_tiles_than_warps(m, interp):
    """400 x 400 pixels are 5000 tiles, more than the device's 3648 warps: the first come back for a second
    one, whose gradients and colour-map sums add to the first's.  Tolerance: as for the small cases of
    test_adjoint_gpu.py."""
    import oracle
    dims, s = (32, 32, 32), 0.02
    cube = scene.diff_cube(dims=dims, n_sources=3)
    cam = scene.orbit_camera(dims, 30, 20, 400, 400)
    lut = scene.linear_lut()
    g = np.random.default_rng(5).normal(size=(400, 400, 4)).astype(np.float32)
    gv, gl, gs = _backward(m, to_dev(cube), cam, to_dev(lut), to_dev(g), s, interp=interp)
    _, rv, rl, rs = oracle.render_grad(cube, cam, g.astype(np.float64), interp=interp, lut=lut, opacity_scale=s)
    assert np.abs(gv.cpu().numpy() - rv).max() <= 1e-4 * np.abs(rv).max()
    assert np.abs(gl.cpu().numpy() - rl).max() <= 1e-4 * np.abs(rl).max()
    assert abs(gs - rs) <= 1e-4 * abs(rs)
