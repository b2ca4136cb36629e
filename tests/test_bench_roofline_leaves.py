"""The upward sweep's traffic in the bench's roofline for leaves that are not 4^3
voxels (a 2x2x2 rule's leaves are 2^3): every leaf gets an expansion, and the M2M
starts from the leaves."""
import argparse
import os
import sys
from types import SimpleNamespace

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def info(leaf_vox):
    """A 6-level tree over a 40^3 block of leaves."""
    L = 6
    hi = [[0, 0, 0] for _ in range(24)]
    for l in range(2, L + 1):
        hi[l] = [-(-40 // (1 << (L - l))) - 1] * 3
    return SimpleNamespace(K=121, L=L, near_pairs=10 ** 8, m2l_pairs=10 ** 5, src_lo=[[0, 0, 0] for _ in range(24)],
                           src_hi=hi, leaf_vox=leaf_vox)


@pytest.mark.parametrize("leaf_vox,top", [(4, 5), (2, 6)])
def test_upward_sweep_traffic(leaf_vox, top):
    args = argparse.Namespace(precision="mixed", p=10, m2l="auto")
    peaks = {"bf16_tflops": 1870.7, "sm_max_mhz": 2070.0, "hbm_gbs": 6700.0}
    nvox = (40 * leaf_vox) ** 3
    ns = {l: (-(-40 // (1 << (6 - l)))) ** 3 for l in range(2, 7)}
    stages = {"eval": 0.1, "m2l": 0.1, "p2m": 0.8, "m2m": 0.7}
    r = bench.fmm_roofline(stages, info(leaf_vox), args, peaks, "w", nvox=nvox, rho_bytes=4)
    assert r["stage"] == "p2m"
    assert r["achieved"] == pytest.approx((4 * nvox + 4 * 121 * ns[top]) / 0.8e-3 / 1e9)
    assert ("p2m_fused" in r["kernel"]) == (leaf_vox != 4)
    r = bench.fmm_roofline(dict(stages, p2m=0.2), info(leaf_vox), args, peaks, "w", nvox=nvox, rho_bytes=4)
    children, parents = sum(ns[l] for l in range(3, top + 1)), sum(ns[l] for l in range(2, top))
    assert r["stage"] == "m2m" and r["achieved"] == pytest.approx(4 * 121 * (children + parents) / 0.7e-3 / 1e9)
