"""Renders from several host threads at once, each on its own stream: requests that share a kernel but
need shared-memory rings of different sizes.  A request that is valid alone must not be refused
because another thread launches the same kernel, and its image must be the one it has alone."""
import ctypes as C
import threading

import numpy as np
import pytest
import torch

import scene
from parity import shw, to_dev

pytestmark = pytest.mark.gpu

ROUNDS = 3000


def _taps(reach):
    return dict(smooth="taps", smooth_taps=(0.5, [float(reach)], [0.25]))


def _axis(dims, W, H, spacing):
    from scene.camera import Camera
    v = lambda *x: np.array(x, np.float32)
    eye = v((dims[0] - 1) / 2 + 0.125, (dims[1] - 1) / 2 - 0.25, -8.0)
    return Camera(eye, v(1, 0, 0), v(0, 1, 0), v(0, 0, 1), 0.0, float(spacing * H / 2), True, W, H)


def _requests(kind):
    """(cube dims, camera, render keywords) of two requests with rings of very different sizes."""
    if kind == "ring":
        d = (68, 64, 66)
        return [(d, scene.orbit_camera(d, 20, 15, 16, 16), _taps(2)), (d, scene.orbit_camera(d, 20, 15, 128, 128), _taps(1))]
    d = (66, 40, 100)
    return [(d, _axis(d, 40, 30, 1.2), {}), (d, _axis(d, 96, 64, 0.25), {})]


@pytest.mark.parametrize("kind", ["ring", "sweep"])
def test_rings_of_different_sizes_in_concurrent_threads(kind):
    m = shw()
    L, api = m._lib.lib(), m.api
    lut = to_dev(scene.linear_lut())
    calls = []
    for dims, cam, kw in _requests(kind) * 2:
        cube = to_dev(scene.tiny_cube(config_id=7, dims=dims, n_sources=2))
        with m.debug_flags("require_staging"):
            want = m.render(cube, cam, "mip", lut=lut, scalar=False, index=False, nsamples=False, **kw)["rgba"]
        calls.append((api.volume_struct(cube), api.camera_struct(cam), api.params_struct("mip", lut, **kw), cube, want,
                      torch.zeros_like(want), torch.cuda.Stream()))
    torch.cuda.synchronize()
    bad, start = [], threading.Barrier(len(calls))

    def work(v, c, p, out, stream):
        start.wait()
        for i in range(ROUNDS):
            s = L.shw_render(C.byref(v), None, C.byref(c), C.byref(p), out.data_ptr(), None, None, None, None, 0,
                             stream.cuda_stream)
            if s != 0:
                bad.append((i, s))
            if i % 16 == 15:
                stream.synchronize()

    with m.debug_flags("require_staging"):
        threads = [threading.Thread(target=work, args=(v, c, p, out, st)) for v, c, p, _, _, out, st in calls]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    torch.cuda.synchronize()
    m.sync_status()
    assert not bad, (len(bad), bad[:3])
    for *_, want, out, _ in calls:
        assert torch.equal(want, out)
