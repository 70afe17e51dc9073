"""The rolling marcher's staging geometry on the host (no GPU): roll_geometry is plain host code,
compiled here with a program that pans views across and past cubes of several shapes.  For every
reach of the taps up to the largest that the API takes it must either refuse the request (the
gather marcher then serves it) or give boxes that hold the sampled footprints in a ring that fits
the shared memory."""
import os
import subprocess


def test_staging_geometry_of_grazing_views(tmp_path):
    from paper_1707_00442_gb300 import build
    src = os.path.join(os.path.dirname(__file__), "roll_geometry.cu")
    exe = str(tmp_path / "roll_geometry")
    # (the kernels are not instantiated; the library's own externals stay unresolved and unused)
    subprocess.run([build.nvcc(), *build._flags(), src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout)
    accepted, refused = map(int, r.stdout.split())
    assert accepted > 1000 and refused > 1000
