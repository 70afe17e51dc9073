"""The rolling marcher (in-ray smoothing from a ring of cube planes in shared memory) on the GPU.

It fetches the gather marcher's corners at the same fixed-point positions and sums the taps in
the same order, so every output must equal the gather marcher's bit for bit (it is forced with
SHW_DEBUG_REQUIRE_STAGING, also where gathering would be faster): views whose major
axis is x, y or z, both directions, parallel and perspective, the eye inside the cube; rows
that are and are not 16-byte multiples, a cube that starts off a 16-byte boundary (bulk copies
of rows); reaches from none to more than the ring holds; cubes smaller than the reach."""
import numpy as np
import pytest
import torch

import scene
from parity import shw, to_dev

pytestmark = pytest.mark.gpu

MODES = ["mip", "avg", "composite", "spectral", "moment1", "composite_spectral", "mip_rgb", "composite_rgb"]
VIEWS = [
    dict(yaw=30, pitch=20, W=100, H=75),                              # z-major
    dict(yaw=100, pitch=10, W=90, H=61),                              # x-major
    dict(yaw=15, pitch=75, W=70, H=83),                               # y-major
    dict(yaw=200, pitch=-35, W=77, H=77),                             # negative directions
    dict(yaw=30, pitch=20, W=160, H=90, ortho=True),                  # parallel
    dict(yaw=-135, pitch=40, W=49, H=33, dist_scale=0.3),             # eye inside the cube
    dict(yaw=0, pitch=0, W=64, H=64, ortho=True),                     # along z
    dict(yaw=250, pitch=-5, W=17, H=9),                               # few, far apart rays
]
DIMS = [(68, 45, 66), (61, 53, 47), (66, 31, 40), (5, 7, 64), (64, 3, 9)]


@pytest.fixture(scope="module")
def m():
    return shw()


def _smooth(m, kind):
    name, n = kind
    if name == "box":
        return dict(smooth="box", smooth_arm=n)
    if name == "wide":  # offsets beyond any ring
        return dict(smooth="taps", smooth_taps=(0.5, [float(n)], [0.25]))
    return dict(smooth="taps", smooth_taps=m.binomial_taps(n, drop=2 if n == 9 else 0))


def _cube(dims, offset):
    c = scene.tiny_cube(config_id=7, dims=dims, n_sources=2)
    c[dims[2] // 3, dims[1] // 2, dims[0] // 4] = np.nan
    flat = torch.empty(c.size + offset, dtype=torch.float32, device="cuda")
    t = flat[offset:].view(c.shape)
    t.copy_(to_dev(c))
    return t


def _same(m, vol, cam, mode, what, **kw):
    lut = to_dev(scene.linear_lut())
    outs = []
    for flags in (("require_staging",), ("no_staging",)):
        try:
            with m.debug_flags(*flags):
                outs.append(m.render(vol, cam, mode, lut=lut, **kw))
                torch.cuda.synchronize()
        except m.ShwError as e:  # a footprint that no ring holds: the default route serves it
            assert e.status == 2 and flags == ("require_staging",)
            outs.append(m.render(vol, cam, mode, lut=lut, **kw))
        m.sync_status()
    for k in outs[0]:
        a, b = outs[0][k].cpu().numpy(), outs[1][k].cpu().numpy()
        assert np.array_equal(a.view(np.int32), b.view(np.int32)), f"{what}: {k}, {(a != b).sum()} of {a.size} differ"


def _cam(dims, v):
    return scene.orbit_camera(dims, v["yaw"], v["pitch"], v["W"], v["H"], ortho=v.get("ortho", False),
                              dist_scale=v.get("dist_scale", 1.0))


@pytest.mark.parametrize("view", range(len(VIEWS)))
@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("kind", [("taps", 9), ("taps", 13), ("box", 2), ("box", 7)])
def test_roll_equals_gather(m, view, dims, kind):
    _same(m, _cube(dims, 0), _cam(dims, VIEWS[view]), "mip", f"{kind} view {view} {dims}", **_smooth(m, kind))


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("kind", [("taps", 5), ("box", 4)])
def test_roll_modes(m, mode, kind):
    kw = dict(opacity_scale=0.3) if mode.startswith("composite") else {}
    dims = (68, 45, 66)
    _same(m, _cube(dims, 0), _cam(dims, VIEWS[0]), mode, f"{mode} {kind}", **kw, **_smooth(m, kind))
    _same(m, _cube(dims, 0), _cam(dims, VIEWS[1]), mode, f"{mode} {kind} clip", filter="clip", min_threshold=-1.0,
          max_threshold=2.0, **kw, **_smooth(m, kind))


@pytest.mark.parametrize("offset", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", [("taps", 9), ("box", 16)])
@pytest.mark.parametrize("dims", [(64, 20, 24), (61, 19, 23)])
def test_roll_unaligned_cubes(m, offset, kind, dims):
    for v in (0, 2, 3):
        _same(m, _cube(dims, offset), _cam(dims, VIEWS[v]), "avg", f"{kind} offset {offset}", **_smooth(m, kind))


@pytest.mark.parametrize("kind", [("wide", 3), ("wide", 12), ("wide", 60), ("taps", 1), ("box", 16)])
@pytest.mark.parametrize("step", [0.5, 0.37])
def test_roll_reaches(m, kind, step):
    dims = (68, 45, 66)
    _same(m, _cube(dims, 0), _cam(dims, VIEWS[0]), "composite", f"{kind} step {step}", step=step, opacity_scale=0.05,
          **_smooth(m, kind))
