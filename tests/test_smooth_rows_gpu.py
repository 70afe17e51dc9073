"""Smoothing by row copies on the GPU: cubes whose rows no tensor copy can take.  The taps are
accumulated in the same order with the same fused multiply-adds as in the kernel without the
pipeline (SHW_DEBUG_SMOOTH_PLAIN), so the results are equal bit for bit: ragged rows, inputs and
outputs that start off a 16-byte boundary, cubes smaller than the radius and than a block, NaN
and infinite voxels, and the interleaved pair form."""
import numpy as np
import pytest
import torch

import oracle
import scene
from parity import TOL_F32, shw, to_dev

pytestmark = pytest.mark.gpu

DIMS = [(61, 43, 47), (66, 41, 40), (67, 33, 5), (1, 1, 1), (2, 3, 2), (5, 70, 9), (33, 2, 3), (101, 31, 64), (131, 75, 11)]


@pytest.fixture(scope="module")
def m():
    return shw()


def _at(shape, offset, src=None):
    flat = torch.full((int(np.prod(shape)) + offset + 4,), 7.0, dtype=torch.float32, device="cuda")
    t = flat[offset:offset + int(np.prod(shape))].view(shape)
    if src is not None:
        t.copy_(to_dev(src))
    return t, flat


def _both(m, fn):
    a = fn()
    with m.debug_flags("smooth_plain"):
        b = fn()
    m.sync_status()
    return a.cpu().numpy().view(np.int32), b.cpu().numpy().view(np.int32)


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("radius", [1, 2, 3, 5, 6, 8])
def test_rows_equal_plain(m, dims, radius):
    cube = scene.tiny_cube(config_id=24, dims=dims, n_sources=2)
    ct = to_dev(cube)
    a, b = _both(m, lambda: m.smooth(ct, radius / 3.0, radius))
    assert np.array_equal(a, b)
    a, b = _both(m, lambda: m.smooth_zip(ct, to_dev(cube + 1), radius / 3.0, radius))
    assert np.array_equal(a, b)


@pytest.mark.parametrize("offsets", [(1, 0), (0, 1), (2, 3), (3, 2), (4, 4)])
@pytest.mark.parametrize("dims", [(64, 20, 24), (61, 19, 23)])
def test_rows_unaligned(m, offsets, dims):
    cube = scene.tiny_cube(config_id=25, dims=dims, n_sources=2)
    cube[3, 4, 5], cube[20, 2, 50] = np.nan, np.inf
    ct, _ = _at(cube.shape, offsets[0], cube)
    out, flat = _at(cube.shape, offsets[1])
    a, b = _both(m, lambda: m.smooth(ct, 1.0, 3, out=out).clone())
    assert np.array_equal(a, b)
    edge = flat.cpu().numpy()  # nothing beside the output is written
    assert (edge[:offsets[1]] == 7.0).all() and (edge[offsets[1] + cube.size:] == 7.0).all()


def test_rows_match_oracle(m):
    cube = scene.tiny_cube(config_id=26, dims=(75, 50, 41), n_sources=2)
    w = np.array([0.1, 0.2, 0.3, 0.25, 0.15], np.float32)  # (an asymmetric kernel as well)
    g = m.smooth_weights(to_dev(cube), w.tolist()).cpu().numpy()
    o = oracle.smooth(cube, w.astype(np.float64))
    assert np.abs(g - o).max() <= TOL_F32 * float(cube.max() - cube.min())
