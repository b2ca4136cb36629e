"""Leaves, ancestors and evaluation items of a plan where their lists span
several tiles of 1,024 (and many more than that): leaves of one observer, of
hundreds, and few of thousands.  The boxes of every level are exact; the field
at a sample of the observers is that of the direct sum (1e-4, some ten times
the degree-8 expansions' truncation; an observer left out would read zero)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("n,m", [((8, 8, 4), 1023), ((8, 8, 4), 5000), ((128, 130, 8), 1025), ((260, 200, 8), 9001),
                                 ((640, 480, 4), 200000), ((640, 480, 4), 2200000)])
def test_lists(n, m):
    xi, w = wl.gauss_rule(1)
    rng = np.random.default_rng(m)
    u = rng.uniform(0.0, 1.0, (m, 2)) ** rng.choice([1.0, 3.0])
    obs = np.concatenate([u * np.array(n[:2], float), np.full((m, 1), n[2] + 0.5)], 1)
    rho = torch.tensor(rng.uniform(0.0, 1.0, n[::-1]), dtype=torch.float32, device=DEV)
    geo = (n, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), xi, w)
    pick = np.concatenate([np.arange(0, m, max(1, m // 200)), [m - 1]])
    with pkg.Plan(*geo, torch.tensor(obs, device=DEV), mode="fmm", precision="mixed", p=8, G=1.0) as plan:
        g = plan.forward(rho)[0].cpu().numpy()
        plan.check()
        keys = plan.export_tree(plan.info.L)[1].astype(np.uint64)
        for level in range(2, plan.info.L + 1):
            boxes = plan.export_tree(level)[2].astype(np.uint64)
            assert np.array_equal(boxes, np.unique(keys >> np.uint64(3 * (plan.info.L - level))))
    with pkg.Plan(*geo, torch.tensor(obs[pick], device=DEV), mode="direct", precision="fp64", G=1.0) as plan:
        ref = plan.forward(rho.double())[0].cpu().numpy()
    assert np.linalg.norm(g[pick] - ref) <= 1e-4 * np.linalg.norm(ref)
    assert np.all(np.any(g != 0.0, axis=-1))
