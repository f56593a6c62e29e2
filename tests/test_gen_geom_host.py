"""The general kernel's block geometry (teams per block, warps per team) on the
host: within the limits of a block for every grid, and the number of warps where
the two choices were measured apart (tests/gen_geom_host.cu). No GPU is needed."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def geom(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = tmp_path_factory.mktemp("geom") / "gen_geom_host"
    src = os.path.join(ROOT, "tests", "gen_geom_host.cu")
    inc = os.path.join(ROOT, "paper_1302_0120_gb300", "csrc")
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I", inc, src, "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lambda *a: subprocess.run([str(exe), *map(str, a)], capture_output=True, text=True, check=True).stdout.strip()


def test_geometry_fits_a_block(geom):
    out = geom()
    assert out.startswith("ok ") and int(out.split()[1]) > 10000, out


@pytest.mark.parametrize("nx,ny,warps", [
    (320, 240, 2), (320, 320, 2), (360, 250, 2), (384, 384, 2), (480, 320, 2),  # four warps 4 to 11 % slower
    (500, 375, 4), (640, 360, 4), (640, 480, 4), (720, 576, 4), (625, 625, 4), (1500, 1500, 4),  # 2 to 9 % faster
    (120, 90, 2), (243, 243, 2), (1280, 1024, 2), (600, 50, 4),
])
def test_warps_per_line(geom, nx, ny, warps):
    assert geom(nx, ny, 1).split()[1] == str(warps)
