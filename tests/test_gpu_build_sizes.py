"""The plan build's sort and scans, and the hexahedral sources, at the sizes
where their tiles end: observers around one and several sort tiles, around the
one-block scan's limit and in the larger tiles; cells around a block's 32 with 1
to 64 nodes.  The sort is exact; the sources' bars are those of the mixed form
(1e-6 of the cell's extent, 1e-6 relative weight)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("m", [1, 31, 255, 257, 2047, 2049, 4097, 262143, 262145, 300001, (4 << 20) - 1, (4 << 20) + 5])
def test_observer_order(m):
    """Stable: ascending keys, ascending indices among equal keys, every index once."""
    n = (64, 48, 32)
    xi, w = wl.gauss_rule(1)
    rng = np.random.default_rng(m)
    obs = np.stack([rng.uniform(0.0, n[0], m), rng.uniform(0.0, n[1], m), np.full(m, float(n[2]) + 1.0)], -1)
    with pkg.Plan(n, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), xi, w, torch.tensor(obs, device=DEV), mode="fmm",
                  precision="mixed", p=4, G=1.0) as plan:
        plan.check()
        perm, keys, boxes, _, _ = plan.export_tree(plan.info.L)
    assert np.array_equal(np.sort(perm), np.arange(m))
    k = keys.astype(np.int64)
    assert np.all(np.diff(k) >= 0)
    assert np.all((np.diff(k) > 0) | (np.diff(perm.astype(np.int64)) > 0))
    assert np.array_equal(np.unique(keys), boxes)


@pytest.mark.parametrize("cells", [(1, 1, 1), (31, 1, 1), (8, 4, 1), (11, 3, 1), (13, 5, 3)])
@pytest.mark.parametrize("npts", [1, 2, 4])
def test_hex_sources_blocks(cells, npts):
    verts = wl.hex_brick_mesh(cells, (4.0e5, 6.2e6, -3000.0), (4.3e5, 6.23e6, 200.0), warp=0.2)
    cell = float(np.ptp(verts, axis=1).max())
    xi, w = wl.gauss_rule(npts)
    x, a = pkg.hex_sources(torch.tensor(verts, device=DEV), xi, w, precision="mixed")
    xr, ar = direct.hex_sources(verts, xi, w)
    assert np.abs(x.cpu().numpy() - xr).max() <= 1e-6 * cell
    assert np.abs(a.cpu().numpy() / ar - 1.0).max() <= 1e-6
