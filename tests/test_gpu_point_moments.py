"""The points' P2M at every lane layout it chooses from (degrees on both sides
of each choice), on leaves that are empty, hold a few points, or enough to take
the whole warp or several segments.

- Against a voxel plan of the same degree on the same sources (a grid's centre
  nodes as points): both fields carry the truncation of leaves of about as many
  sources, so the points' error may be at most 4 times the voxels' (plus 1e-12
  or, in mixed precision, 2e-6 for rounding).
- A point split into equal coincident parts: its plan's leaves are other ones
  (more points), its field is the same, so its error against the oracle may be
  at most 4 times the unsplit plan's (plus 1e-11 or 2e-6).
- Batch members against the same density alone: 1e-12 or 2e-6 (the M2L's tiles
  differ between the two)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def t(a, dt=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dt, device=DEV)


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p", [3, 6, 7, 8, 9, 10, 12, 13, 15, 16])
def test_against_voxels_of_the_same_degree(p, precision):
    n = (24, 20, 22)
    wk = wl.random_small(500 + p, n=n, n_obs=300, h=(1.0, 1.0, 1.0), origin=(2.0, -9.0, -30.0), obs_pad=2.0)
    rho = wk.rho.astype(np.float32).astype(np.float64)
    xi, w = wl.gauss_rule(1)
    ref = direct.forward(n, wk.grid.origin, wk.grid.h, xi, w, rho, wk.obs, 1.0)
    ax = [wk.grid.origin[d] + (np.arange(n[d]) + 0.5) * wk.grid.h[d] for d in range(3)]
    x = np.stack(np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")[::-1], -1).reshape(-1, 3)
    a = np.full(len(x), float(np.prod(wk.grid.h)))
    dt = torch.float32 if precision == "mixed" else torch.float64
    kw = dict(mode="fmm", precision=precision, p=p, G=1.0)
    with pkg.Plan(n, wk.grid.origin, wk.grid.h, xi, w, t(wk.obs), **kw) as plan:
        vox = rel_l2(plan.forward(t(rho, dt))[0].cpu().numpy().reshape(-1, 3), ref)
    with pkg.PointsPlan(t(x), t(a), t(wk.obs), **kw) as plan:
        pts = rel_l2(plan.forward(t(rho.ravel(), dt))[0].cpu().numpy(), ref)
        plan.check()
    print("p %d %s: voxels %.2e points %.2e" % (p, precision, vox, pts))
    assert pts <= 4 * vox + (2e-6 if precision == "mixed" else 1e-12)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p", [5, 9, 12, 16])
def test_points_per_leaf(p, precision):
    rng = np.random.default_rng(40 + p)
    cl = rng.uniform(0.0, 64.0, (400, 3))
    x = np.concatenate([rng.uniform(0.0, 64.0, (3000, 3)), cl])
    a = rng.uniform(0.5, 1.5, len(x))
    parts = np.ones(len(x), dtype=np.int64)
    parts[3000:3020] = [2, 17, 200, 255, 256, 257, 300, 511, 700, 1023, 1024, 1025, 1300, 2047, 2048, 2049, 2500, 3001, 3, 1]
    xs, ws = np.repeat(x, parts, axis=0), np.repeat(a / parts, parts)
    obs = rng.uniform(-20.0, 84.0, (500, 3))
    dt = torch.float32 if precision == "mixed" else torch.float64
    rho = rng.normal(size=(2, len(x))).astype(np.float32).astype(np.float64)
    out = []
    for xx, ww, rr in ((x, a, rho), (xs, ws, np.repeat(rho, parts, axis=1))):
        with pkg.PointsPlan(t(xx), t(ww), t(obs), mode="fmm", precision=precision, p=p, max_batch=2, G=1.0) as plan:
            both = plan.forward(t(rr, dt))[0].cpu().numpy()
            for b in range(2):
                one = plan.forward(t(rr[b], dt))[0].cpu().numpy()
                assert rel_l2(one, both[b]) <= (2e-6 if precision == "mixed" else 1e-12)
            out.append(both)
    ref = np.stack([direct.forward_points(x, a, 1, rho[b], obs, 1.0) for b in range(2)])
    e0, e1 = rel_l2(out[0], ref), rel_l2(out[1], ref)
    print("p %d %s: whole %.2e split %.2e" % (p, precision, e0, e1))
    assert e1 <= 4 * e0 + (2e-6 if precision == "mixed" else 1e-11)
