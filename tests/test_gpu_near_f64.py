"""The FP64 near and far field of rules on a 4^3 lattice per leaf (one node in
4^3-voxel leaves, 2^3 nodes in 2^3-voxel leaves), and the general form beside it,
against the FP64 oracle: observers on the nodes themselves, on voxel faces, edges
and corners, scattered around, few and many to a leaf, in batches and source parts.
Bar: the FP64 FMM's (1e-6 at p >= 14)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("npts,p", [(1, 14), (2, 14), (3, 14), (1, 16)])
def test_positions(npts, p):
    n = (19, 14, 17)
    rng = np.random.default_rng(npts)
    xi, w = wl.gauss_rule(npts)
    rho = rng.normal(size=n[::-1])
    ax = [np.arange(0.0, n[d] + 0.1, 0.5) for d in range(3)]
    lat = np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)     # centres, faces, edges, corners
    obs = np.concatenate([lat[rng.permutation(len(lat))[:3000]], rng.uniform(-3.0, np.array(n) + 3.0, (1500, 3)),
                          rng.uniform(4.0, 8.0, (300, 3))])
    origin, h = (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)
    ref = direct.forward(n, origin, h, xi, w, rho, obs, 1.0)
    r = torch.tensor(np.stack([rho, -2.0 * rho]), device=DEV)
    with pkg.Plan(n, origin, h, xi, w, torch.tensor(obs, device=DEV), mode="fmm", precision="fp64", p=p, G=1.0,
                  max_batch=2) as plan:
        g = plan.forward(r)[0].cpu().numpy()
        plan.check()
        print("npts %d p %d: %.2e" % (npts, p, rel_l2(g[0], ref)))
        assert rel_l2(g[0], ref) <= 1e-6
        assert np.array_equal(g[1], -2.0 * g[0])
        assert np.array_equal(plan.forward(r[0])[0].cpu().numpy(), g[0])
        parts = np.zeros_like(g[0])
        for part in range(3):
            plan.set_source_part(part, 3)
            parts += plan.forward(r[0])[0].cpu().numpy()
        assert rel_l2(parts, ref) <= 1e-6
