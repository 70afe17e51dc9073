"""The plane sweep's staged box on the host (no GPU): for every pixel footprint, up to views so far
zoomed out that a tile spans more voxels than an int holds, the box either is refused (the general
marcher then serves the request) or holds the footprint within the copies' and the ring's limits."""
import os
import subprocess


def test_staged_box_of_every_footprint(tmp_path):
    from paper_1707_00442_gb300 import build
    src = os.path.join(os.path.dirname(__file__), "axis_box.cu")
    exe = str(tmp_path / "axis_box")
    subprocess.run([build.nvcc(), *build._flags(), src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stdout)
    accepted, refused = map(int, r.stdout.split())
    assert accepted > 1000 and refused > 1000
