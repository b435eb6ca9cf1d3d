"""Slices of a batch that differ in path or filter meet in the operators they
share (CPU): one launch for each distinct operator of a step."""
import glob
import os
import subprocess

import pytest

from paper_1310_1434_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
K, I = 30, 8
COMMON = {"FIN", "ZERO", "RESTART"}, {"FIN", "CG_A"}


def operators(form):
    """Grouped operators of a slice: of the prologue, and of a CG step."""
    orb, tc = form[0] == "1", form[1] == "1"
    ops = {"ORB_BWD" if orb else "BWD"} | (set() if tc else {"RAMP"}) | ({"ORB_ZPACK"} if orb and tc else set())
    step = {"ORB_PACK", "ORB_FWD"} if orb else {"TRANSPOSE", "FWD", "CG_B"}
    return ops | COMMON[0], ops | COMMON[1] | step


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    build.build()
    exe = str(tmp_path_factory.mktemp("batch") / "batch_programs")
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    r = subprocess.run([build._nvcc(), "-std=c++17", "-O2", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH +
                       [os.path.join(HERE, "batch_programs.cu")] + objs + ["-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("forms", [["10"], ["11"], ["00"], ["01"], ["10", "11"], ["11", "01"], ["00", "01"],
                                   ["10", "00"], ["10", "01"], ["11", "00"], ["10", "11", "00", "01"]],
                         ids="+".join)
def test_one_launch_for_each_operator(program, forms):
    r = subprocess.run([program, str(K), str(I)] + forms, capture_output=True, text=True)
    assert r.returncode == 0
    prologue, step = (set.union(*(operators(f)[i] for f in forms)) for i in (0, 1))
    assert int(r.stdout) == len(prologue) + K * I * len(step) + K + K - 1      # and SHRINK, RESTART
