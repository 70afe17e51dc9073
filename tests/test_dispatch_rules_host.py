"""Where each staged or widened form is taken, on the host (no GPU): the rules are plain host code, compiled
here and asked about requests whose two routes were measured.  Every time is microseconds on a
GB300, of the route named first and of the other; the rule must take the faster."""
import os
import subprocess

import pytest

import scene
from scene.camera import ortho_axis_camera


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    from paper_1707_00442_gb300 import build
    src = os.path.join(os.path.dirname(__file__), "dispatch_rules.cu")
    exe = str(tmp_path_factory.mktemp("rules") / "dispatch_rules")
    subprocess.run([build.nvcc(), *build._flags(), src, "-o", exe], check=True)

    def run(rule, dims, cam, k=0):
        v = [*cam.eye, *cam.right, *cam.up, *cam.fwd, cam.tan_half_fovy, cam.ortho_half_h]
        line = " ".join([rule, *(repr(float(x)) for x in v),
                         *(str(int(x)) for x in (cam.ortho, cam.width, cam.height, *dims, k))])
        r = subprocess.run([exe], input=line, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stderr
        return int(r.stdout)
    return run


@pytest.mark.parametrize("dims,yaw,W,H,more,plain", [
    ((50, 50, 37), 70, 1000, 1000, 204, 240), ((750, 750, 70), 20, 1000, 1000, 333, 446),
    ((301, 300, 300), 30, 1600, 1600, 2583, 2871),
    ((641, 641, 641), 0, 500, 500, 1088, 1496), ((641, 641, 641), 70, 1000, 1000, 5560, 4870),
    ((65, 66, 67), 30, 64, 64, 75, 58), ((201, 200, 200), 0, 200, 200, 210, 165),
    ((68, 388, 169), 227, 169, 549, 433, 321), ((419, 52, 107), 172, 132, 753, 113, 81)])
def test_more_resident_ctas(ask, dims, yaw, W, H, more, plain):
    """Gathered ratios of two cubes, the second compositing: compiled for more resident CTAs, and not."""
    assert ask("many", dims, scene.orbit_camera(dims, yaw, 20, W, H)) == (more < plain)


def test_more_resident_ctas_counts_pixels_of_the_image(ask):
    """Views that show part of a wide cube: 156 and 103 us, 122 and 88."""
    assert not ask("many", (332, 44, 149), scene.orbit_camera((332, 44, 149), 182.22, -10.72, 396, 892))
    assert not ask("many", (560, 73, 123), scene.orbit_camera((560, 73, 123), 173.62, 9.86, 182, 1095))


@pytest.mark.parametrize("dims,yaw,pitch,W,staged,gathered", [
    ((512, 512, 512), 85, 10, 1000, 2422, 3959), ((256, 256, 256), 60, -30, 400, 238, 425),
    ((64, 64, 512), 60, -30, 400, 75, 131), ((1024, 1024, 1024), 55, 20, 500, 2808, 4938),
    ((512, 512, 512), 70, 20, 640, 1640, 1713),
    ((200, 200, 200), 85, 10, 256, 495, 189), ((512, 512, 512), 85, 10, 256, 2483, 856),
    ((48, 48, 48), 85, 10, 1000, 165, 149)])
def test_staged_marcher(ask, dims, yaw, pitch, W, staged, gathered):
    """MIP of a float32 cube: the staged marcher, and the gather."""
    assert ask("staged", dims, scene.orbit_camera(dims, yaw, pitch, W, W)) == (staged < gathered)


@pytest.mark.parametrize("rule,dims,yaw,pitch,W,staged,gathered", [
    ("staged", (64, 64, 512), 60, -30, 128, 151, 62), ("staged", (256, 256, 64), 20, 60, 128, 189, 87),
    ("staged_composite", (512, 512, 512), 60, -30, 1000, 1381, 2952),
    ("staged_composite", (128, 512, 256), 45, 45, 1000, 496, 1045),
    ("staged_composite", (512, 128, 128), 85, 10, 128, 1190, 255)])
def test_staged_marcher_of_few_tiles(ask, rule, dims, yaw, pitch, W, staged, gathered):
    """Coarse views of few tiles, which a gather spreads over more SMs, and compositing."""
    assert ask(rule, dims, scene.orbit_camera(dims, yaw, pitch, W, W)) == (staged < gathered)


def test_staged_marcher_of_few_tiles_by_their_pitch(ask):
    """An average at 2.03 voxels per pixel: 114 us staged, 150 gathered."""
    cam = scene.orbit_camera((96, 87, 204), 55.38, 10.57, 740, 119, ortho=True)
    assert ask("staged", (96, 87, 204), cam)


def test_staged_marcher_of_pairs(ask):
    for dims, yaw, pitch, W, staged, gathered in [((64, 64, 512), 60, -30, 640, 129, 161),
                                                  ((256, 256, 256), 85, 10, 256, 965, 420)]:
        assert ask("staged_pair", dims, scene.orbit_camera(dims, yaw, pitch, W, W)) == (staged < gathered)


MIP, COMPOSITE, MOMENT1 = 0, 2, 5


@pytest.mark.parametrize("rule,n,nz,mode,rows,gathered", [
    ("rows", 350, 454, MIP, 296, 749), ("rows", 601, 300, MIP, 459, 958), ("rows", 601, 300, COMPOSITE, 636, 789),
    ("rows", 71, 300, COMPOSITE, 213, 151), ("rows", 65, 97, MOMENT1, 98, 72), ("rows", 131, 400, MOMENT1, 340, 275),
    ("rows_nearest", 601, 300, MIP, 440, 595), ("rows_nearest", 65, 97, MIP, 80, 54),
    ("rows_nearest", 131, 400, MIP, 271, 187), ("rows_nearest", 401, 20, COMPOSITE, 74, 52)])
def test_sweep_by_row_copies(ask, rule, n, nz, mode, rows, gathered):
    """Spectral-axis views of n x n x nz cubes, one pixel a voxel: the sweep by row copies, and the gather."""
    assert ask(rule, (n, n, nz), ortho_axis_camera((n, n, nz), n, n), mode) == (rows < gathered)


def test_sweep_by_row_copies_of_magnified_views(ask):
    for n, nz, W, mode, rows, gathered in [(71, 300, 142, MIP, 166, 209), (131, 97, 262, COMPOSITE, 113, 128)]:
        assert ask("rows", (n, n, nz), ortho_axis_camera((n, n, nz), W, W), mode) == (rows < gathered)


@pytest.mark.parametrize("rule,dims,yaw,pitch,W,ring,gathered", [
    ("taps", (512, 512, 512), 100, 10, 1000, 7873, 82899), ("taps", (512, 512, 512), 30, 20, 1000, 8656, 24064),
    ("taps", (160, 160, 160), 100, 10, 500, 941, 3855), ("taps_composite", (512, 512, 512), 30, 20, 1000, 6667, 16482),
    ("taps_composite", (512, 512, 512), 20, 75, 1000, 7446, 7167), ("taps", (129, 129, 129), 15, 20, 128, 802, 483),
    ("taps_composite", (68, 512, 68), 20, 75, 128, 2751, 685), ("taps_composite", (64, 64, 512), 15, 20, 128, 2466, 722),
    ("box", (512, 512, 512), 100, 10, 1000, 2356, 8305), ("box_composite", (512, 512, 512), 100, 10, 1000, 1820, 4474),
    ("box", (400, 70, 400), 60, -30, 500, 705, 267), ("box_composite", (320, 320, 320), 15, 20, 128, 718, 264),
    ("box_composite", (512, 512, 512), 20, 75, 1000, 2265, 2163)])
def test_rolling_marcher(ask, rule, dims, yaw, pitch, W, ring, gathered):
    """9 taps, or the box of 3 to 9: the ring, and the gather."""
    assert ask(rule, dims, scene.orbit_camera(dims, yaw, pitch, W, W), 2) == (ring < gathered)


@pytest.mark.parametrize("rule,dims,yaw,pitch,W,ring,gathered", [
    ("taps", (64, 64, 512), 100, 10, 500, 426, 3336), ("taps", (400, 70, 400), 100, 10, 500, 1245, 4965),
    ("taps_composite", (512, 512, 512), 100, 10, 500, 4151, 16966),
    ("box", (512, 512, 512), 0, 0, 500, 682, 1178), ("box", (240, 240, 240), 60, -30, 500, 444, 592),
    ("box_composite", (512, 512, 512), 60, -30, 1000, 2241, 4109)])
def test_rolling_marcher_where_a_warp_gathers_many_rows(ask, rule, dims, yaw, pitch, W, ring, gathered):
    cam = scene.orbit_camera(dims, yaw, pitch, W, W, ortho=(yaw == 0))
    assert ask(rule, dims, cam, 2) == (ring < gathered)
