"""The bounds-checked build (-DSHW_CHECKED) through the marchers that stage planes in rings of their own
layout: in-ray smoothing (taps and box; views whose major axis is x, y and z; rows that tensor
copies take and rows that they do not) and the spectral-axis sweep by row copies, in both
directions.  The staged form is forced, so a refusal fails the test; no check may record a
violation and every output must be the normal library's."""
import pytest

import scene
from parity import to_dev
from test_axis_rows_gpu import _cam as axis_cam
from test_axis_rows_gpu import _cube as axis_cube
from test_roll_gpu import VIEWS, _cam, _cube, _smooth
from test_zz_checked_gpu import _both, libs  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


def _forced(m, *args, **kw):
    with m.debug_flags("require_staging"):
        return m.render(*args, lut=to_dev(scene.linear_lut()), **kw)


@pytest.mark.parametrize("view", range(7))
@pytest.mark.parametrize("dims,offset", [((68, 45, 66), 0), ((61, 53, 47), 0), ((64, 20, 24), 1)])
@pytest.mark.parametrize("kind", [("taps", 9), ("box", 2)])
def test_checked_ring(libs, view, dims, offset, kind):  # noqa: F811
    m = libs[0]
    vol, cam = _cube(dims, offset), _cam(dims, VIEWS[view])
    _both(libs, lambda: _forced(m, vol, cam, "mip", **_smooth(m, kind)))


@pytest.mark.parametrize("dims,offset", [((61, 43, 47), 0), ((66, 41, 40), 0), ((64, 20, 24), 3), ((2, 3, 2), 0)])
@pytest.mark.parametrize("view", [(100, 70, 0.75, False), (37, 29, 1.0, True)])
def test_checked_row_sweep(libs, dims, offset, view):  # noqa: F811
    m = libs[0]
    W, H, spacing, down = view
    vol, cam = axis_cube(dims, offset), axis_cam(dims, W, H, spacing, down)
    for mode in ("mip", "composite", "moment1"):
        _both(libs, lambda mode=mode: _forced(m, vol, cam, mode))
