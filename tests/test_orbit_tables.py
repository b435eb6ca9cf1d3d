"""The orbit tables against the general ray table, on the CPU (tests/orbit_tables.cu
says what is compared): every group of symmetries, odd and even sides and bin
counts, ragged tiles, views that a mirror takes to themselves, and scans that
have to be left to the general path."""
import glob
import math
import os
import subprocess

import pytest

from paper_1310_1434_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    build.build()
    exe = str(tmp_path_factory.mktemp("orbit") / "orbit_tables")
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    r = subprocess.run([build._nvcc(), "-std=c++17", "-O2", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH +
                       [os.path.join(HERE, "orbit_tables.cu")] + objs + ["-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("n,px,V,nb,dso,beta0,frames", [
    (64, 1.1, 16, 64, 850.0, 0.0, 8),                 # mirrors and quarter turns
    (77, 1.3, 32, 101, 850.0, 0.0, 8),                # odd bins: orbits that hold a ray twice
    (97, 1.1, 36, 64, 850.0, 0.0, 8),                 # V = 4 mod 8, fewer rays than pixels
    (66, 1.0, 20, 95, 850.0, math.pi / 20, 8),        # the mirror between two views
    (65, 1.1, 18, 91, 850.0, 0.0, 4),                 # mirrors and a half turn: two classes
    (70, 1.1, 20, 101, 850.0, 0.2, 4),                # quarter turns alone: two classes
    (64, 6.4, 60, 92, 850.0, 0.0, 8),                 # coarse pixels: a strongly curved fan
    (72, 1.0, 24, 180, 850.0, 0.0, 8),                # two rays a pixel
    (66, 1.0, 40, 101, 850.0, 0.0, 0),                # a ray along a grid line
    (70, 1.0, 24, 130, 60.0, 0.0, 0),                 # source too close
    (77, 1.3, 31, 101, 850.0, 0.0, 0),                # a mirror alone
    (70, 1.3, 30, 101, 850.0, 0.1, 0),                # a half turn alone
    (63, 1.1, 16, 64, 850.0, 0.0, 0),                 # small image
    (64, 1.0, 16, 1024, 850.0, 0.0, 0),               # rays much denser than pixels
])
def test_orbits_match_the_general_table(program, n, px, V, nb, dso, beta0, frames):
    r = subprocess.run([program] + [repr(a) for a in (n, px, V, nb, dso, beta0)], capture_output=True, text=True)
    assert r.returncode == 0, r.returncode
    assert int(r.stdout) == frames
