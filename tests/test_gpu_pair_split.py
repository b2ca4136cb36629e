"""Direct sums whose sources are split over the warps of a cluster: observer
counts around the 32- and 64-observer tiles, rows around the 30-voxel piece,
and fewer sources than warps, against the FP64 oracle.  Bars as for every
direct sum: 1e-12 in FP64, 1e-5 in mixed precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("m", [1, 32, 33, 64, 65, 200])
@pytest.mark.parametrize("n,npts", [((1, 1, 1), 1), ((30, 2, 1), 1), ((31, 1, 3), 2), ((61, 5, 2), 1), ((2, 3, 90), 2)])
def test_direct_split_edges(n, npts, m):
    wk = wl.random_small(40 + m, n=n, npts=npts, n_obs=m, B=2)
    ref = direct.forward(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, wk.rho, wk.obs, wk.G)
    obs = torch.tensor(wk.obs, dtype=torch.float64, device=DEV)
    rho = torch.tensor(wk.rho, device=DEV)
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):
        with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, mode="direct", precision=prec,
                      max_batch=2, G=wk.G) as plan:
            g, gz = plan.forward(rho, want_gz=True)
            again, _ = plan.forward(rho)
            assert rel_l2(g.cpu().numpy(), ref) <= tol
            assert torch.equal(gz, g[..., 2]) and torch.equal(g, again)


@pytest.mark.parametrize("m", [1, 32, 33, 150])
def test_closed_form_split_edges(m):
    wk = wl.random_small(60 + m, n=(5, 1, 3), n_obs=m, h=(1.0, 1.0, 1.0))
    ref = direct.forward_analytic(wk.grid.n, wk.grid.origin, wk.grid.h, wk.rho, wk.obs, wk.G)
    obs = torch.tensor(wk.obs, dtype=torch.float64, device=DEV)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, mode="direct", precision="fp64",
                  voxels="closed_form", G=wk.G) as plan:
        g, _ = plan.forward(torch.tensor(wk.rho, device=DEV))
        assert rel_l2(g.cpu().numpy(), ref) <= 1e-12


@pytest.mark.parametrize("m", [1, 64, 65])
@pytest.mark.parametrize("s", [1, 31, 257, 2000])
def test_points_split_edges(s, m):
    rng = np.random.default_rng(70 + s + m)
    x = rng.uniform(-50.0, 50.0, size=(s, 3))
    a, rho = rng.uniform(0.5, 2.0, size=s), rng.normal(2500.0, 300.0, size=s)
    obs = rng.uniform(-70.0, 70.0, size=(m, 3))
    obs[0] = x[0]   # a coincident pair contributes nothing
    ref = direct.forward_points(x, a, 1, rho, obs, 1.0)
    t = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)  # noqa: E731
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):
        with pkg.PointsPlan(t(x), t(a), t(obs), mode="direct", precision=prec, G=1.0) as plan:
            g = plan.forward(t(rho))[0].cpu().numpy()
            assert np.linalg.norm(g - ref) <= tol * np.linalg.norm(ref)   # 0 <= 0 for the lone coincident pair
