"""The staged forms of in-ray smoothing, the spectral-axis sweep and the separable smoothing must be
the ones that run: every request here is made with the forms that would stand in for them switched
off, and a refusal fails the test (the requests that no ring holds must be refused).  Outputs equal
the gather marcher's, or the plain smoothing kernel's, bit for bit."""
import numpy as np
import pytest
import torch

import scene
from parity import shw, to_dev
from test_axis_rows_gpu import _cam as axis_cam
from test_axis_rows_gpu import _cube as axis_cube
from test_roll_gpu import VIEWS, _cam, _cube, _smooth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    return shw()


def _render(m, flags, vol, cam, mode, **kw):
    with m.debug_flags(*flags):
        out = m.render(vol, cam, mode, lut=to_dev(scene.linear_lut()), **kw)
        torch.cuda.synchronize()
    m.sync_status()
    return {k: v.cpu().numpy().view(np.int32) for k, v in out.items()}


def _served(m, other, vol, cam, mode, **kw):
    a, b = _render(m, ("require_staging",), vol, cam, mode, **kw), _render(m, other, vol, cam, mode, **kw)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("view", range(7))
@pytest.mark.parametrize("dims,offset", [((68, 45, 66), 0), ((61, 53, 47), 0), ((66, 31, 40), 0), ((5, 7, 64), 0),
                                         ((64, 20, 24), 1), ((61, 19, 23), 3)])
@pytest.mark.parametrize("kind", [("taps", 9), ("wide", 3), ("box", 2), ("box", 16)])
def test_ring_serves(m, view, dims, offset, kind):
    _served(m, ("no_staging",), _cube(dims, offset), _cam(dims, VIEWS[view]), "composite", opacity_scale=0.05,
            **_smooth(m, kind))


@pytest.mark.parametrize("view,kind", [(0, ("wide", 12)), (2, ("wide", 60)), (7, ("box", 2))])
def test_ring_refuses(m, view, kind):
    dims = (68, 45, 66)
    with pytest.raises(m.ShwError) as e:
        _render(m, ("require_staging",), _cube(dims, 0), _cam(dims, VIEWS[view]), "mip", **_smooth(m, kind))
    assert e.value.status == 2


@pytest.mark.parametrize("dims,offset", [((61, 43, 47), 0), ((66, 41, 40), 0), ((65, 44, 5), 0), ((7, 5, 90), 0),
                                         ((301, 30, 9), 0), ((64, 20, 24), 1), ((62, 21, 25), 3)])
@pytest.mark.parametrize("mode", ["mip", "composite", "moment1"])
@pytest.mark.parametrize("view", [(100, 70, 0.75, False), (37, 29, 1.0, True), (200, 150, 0.4, False)])
def test_sweep_serves_ragged_rows(m, dims, offset, mode, view):
    W, H, spacing, down = view
    kw = dict(opacity_scale=0.1) if mode == "composite" else {}
    _served(m, ("no_axis_sweep",), axis_cube(dims, offset), axis_cam(dims, W, H, spacing, down), mode, **kw)


@pytest.mark.parametrize("dims", [(131, 95, 21), (97, 99, 40)])  # 15 and 16 blocks: the row copies at every radius
@pytest.mark.parametrize("radius", range(1, 9))
def test_ragged_smoothing_of_many_blocks(m, dims, radius):
    cube = scene.tiny_cube(config_id=24, dims=dims, n_sources=2)
    ct, first = to_dev(cube), to_dev(cube + 1)

    def both():
        return [x.cpu().numpy().view(np.int32) for x in (m.smooth(ct, radius / 3.0, radius),
                                                         m.smooth_zip(ct, first, radius / 3.0, radius))]
    a = both()
    with m.debug_flags("smooth_plain"):
        b = both()
    m.sync_status()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
