"""The FP32 near field of closed-form voxels against the FP64 oracle with the
observers where its forms change: on voxel faces, edges and corners (zero
coordinates of the corner function), inside voxels, around and above the grid,
more and fewer than a warp of them to a leaf, with empty voxels and source parts.
Bar: the mixed-precision FMM's (1e-5)."""
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


def observers(kind, n, rng):
    if kind == "lattice":      # faces, edges, corners and centres in and around the grid
        ax = [np.arange(-2.0, n[d] + 2.5, 0.5) for d in range(3)]
        g = np.stack(np.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)
        return g[rng.permutation(len(g))[:5000]]
    if kind == "stations":     # dense over the top: many warps to a leaf
        x, y = np.meshgrid(np.linspace(0.1, n[0] - 0.1, 150), np.linspace(0.1, n[1] - 0.1, 150))
        return np.stack([x.ravel(), y.ravel(), np.full(x.size, n[2] + 0.25)], -1)
    return rng.uniform(-3.0, np.array(n) + 3.0, (3000, 3))


@pytest.mark.parametrize("kind", ["lattice", "stations", "random"])
@pytest.mark.parametrize("holes", [False, True])
def test_against_the_oracle(kind, holes):
    n = (22, 17, 19)
    rng = np.random.default_rng(7)
    rho = rng.normal(size=n[::-1]).astype(np.float32)
    if holes:
        rho[rng.uniform(size=rho.shape) < 0.4] = 0.0
        rho[5:9] = 0.0
    obs = observers(kind, n, rng)
    origin, h = (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)
    xi, w = wl.gauss_rule(1)
    ref = direct.forward_analytic(n, origin, h, rho.astype(np.float64), obs, 1.0)
    r = torch.tensor(rho, device=DEV)
    with pkg.Plan(n, origin, h, xi, w, torch.tensor(obs, device=DEV), mode="fmm", precision="mixed", p=14, G=1.0,
                  voxels="closed_form") as plan:
        g = plan.forward(r)[0].cpu().numpy()
        plan.check()
        print("%s holes %d: rel L2 %.2e" % (kind, holes, rel_l2(g, ref)))
        assert rel_l2(g, ref) <= 1e-5
        assert np.array_equal(g, plan.forward(r)[0].cpu().numpy())
        parts = np.zeros_like(g)
        for part in range(2):
            plan.set_source_part(part, 2)
            parts += plan.forward(r)[0].cpu().numpy()
        assert rel_l2(parts, ref) <= 1e-5
