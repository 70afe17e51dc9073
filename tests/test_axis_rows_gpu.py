"""The plane sweep by row copies on the GPU: spectral-axis views of cubes whose rows no tensor copy
can take.  It takes the general marcher's samples, so every output must equal the general
marcher's bit for bit: each residue of the row and plane pitches and of the cube's start modulo
16 bytes, both directions, every mode, boxes that reach past the cube, more planes than the ring
holds and fewer, the smallest cubes (SHW_DEBUG_REQUIRE_STAGING forces the sweep where gathering
would be as fast)."""
import numpy as np
import pytest
import torch

import scene
from parity import shw, to_dev

pytestmark = pytest.mark.gpu

DIMS = [(61, 43, 47), (66, 41, 40), (67, 40, 33), (65, 44, 5), (7, 5, 90), (2, 3, 2), (3, 2, 1), (301, 30, 9)]


@pytest.fixture(scope="module")
def m():
    return shw()


def _cube(dims, offset=0):
    c = scene.tiny_cube(config_id=7, dims=dims, n_sources=2)
    c[dims[2] // 3, dims[1] // 2, dims[0] // 4] = np.nan
    flat = torch.empty(c.size + offset, dtype=torch.float32, device="cuda")
    t = flat[offset:].view(c.shape)
    t.copy_(to_dev(c))
    return t


def _cam(dims, W, H, spacing, down=False):
    nx, ny, nz = dims
    f = -1.0 if down else 1.0
    eye = np.array([(nx - 1) / 2 + 0.125, (ny - 1) / 2 - 0.25, nz + 8.0 if down else -8.0])
    v = lambda *x: np.array(x, np.float32)
    return scene.Camera(v(*eye), v(1, 0, 0), v(0, 1, 0), v(0, 0, f), 0.0, float(spacing * H / 2), True, W, H)


def _same(m, vol, cam, mode, what, **kw):
    lut = to_dev(scene.linear_lut())
    outs = []
    for flags in (("require_staging",), ("no_axis_sweep",)):
        try:
            with m.debug_flags(*flags):
                outs.append(m.render(vol, cam, mode, lut=lut, **kw))
                torch.cuda.synchronize()
        except m.ShwError as e:  # a box too wide for the ring: the default route serves it
            assert e.status == 2 and flags == ("require_staging",)
            outs.append(m.render(vol, cam, mode, lut=lut, **kw))
        m.sync_status()
    assert int(outs[0]["nsamples"].max()) > 0, what
    for k in outs[0]:
        a, b = outs[0][k].cpu().numpy(), outs[1][k].cpu().numpy()
        assert np.array_equal(a.view(np.int32), b.view(np.int32)), f"{what}: {k}, {(a != b).sum()} of {a.size} differ"


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("interp", ["trilinear", "nearest"])
@pytest.mark.parametrize("view", [(100, 70, 0.75, False), (37, 29, 2.0, True), (200, 150, 0.4, False)])
def test_rows_sweep_equals_general(m, dims, interp, view):
    W, H, spacing, down = view
    _same(m, _cube(dims), _cam(dims, W, H, spacing, down), "mip", f"{dims} {interp} {view}", interp=interp)


@pytest.mark.parametrize("mode", ["mip", "avg", "composite", "spectral", "moment1"])
@pytest.mark.parametrize("step", [0.5, 1.0, 0.37])
def test_rows_sweep_modes(m, mode, step):
    kw = dict(opacity_scale=0.3) if mode == "composite" else {}
    for dims, down in ((DIMS[0], False), (DIMS[1], True)):
        _same(m, _cube(dims), _cam(dims, 100, 70, 0.75, down), mode, f"{mode} {dims} {step}", step=step, **kw)


@pytest.mark.parametrize("offset", [1, 2, 3, 4])
@pytest.mark.parametrize("dims", [(64, 20, 24), (61, 19, 23), (62, 21, 25)])
def test_rows_sweep_unaligned(m, offset, dims):
    _same(m, _cube(dims, offset), _cam(dims, 90, 40, 0.8), "avg", f"{dims} offset {offset}")
