"""The folded translations rest on the mirror symmetry of the operators: a
host build of the library's own operator entries (fmm_math.cuh) checks every
entry of M2M, M2L and L2L at every mirrored position, and the triangles."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("p", [1, 2, 5, 8])
def test_operators_are_mirror_images(p, tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "mirror_ops")
    subprocess.run([cxx, "-O1", "-std=c++17", "-x", "c++", os.path.join(ROOT, "tests", "emu", "mirror_ops.cpp"),
                    "-I" + os.path.join(ROOT, "paper_1107_5951_gb300", "csrc"), "-o", exe], check=True)
    m2m, m2l, l2l, outside = map(float, subprocess.run([exe, str(p)], check=True, capture_output=True,
                                                       text=True).stdout.split())
    # entries are at most about 1; both sides come from the same recursions
    assert max(m2m, m2l, l2l) <= 1e-14
    assert outside == 0.0
