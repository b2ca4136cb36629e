"""Direct sums of few sources over many observers, where a warp takes a tile of
observers by itself: against the FP64 oracle at the direct sums' bars (1e-12 in FP64,
1e-5 mixed), for rows along each axis, tile edges, a coincident pair, batches; and a
million observers of one voxel take no more than four times a plain copy of that many
fields (the sums' sharing among blocks took twenty times)."""
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


def dev(a):
    return torch.tensor(a, dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("m", [50000, 50017])
@pytest.mark.parametrize("n,npts", [((1, 1, 1), 1), ((1, 1, 64), 1), ((2, 61, 1), 1), ((3, 2, 4), 2), ((31, 1, 2), 1)])
def test_voxels(n, npts, m):
    wk = wl.random_small(50 + m % 7, n=n, npts=npts, n_obs=m, B=2)
    wk.obs[m - 1] = np.array(wk.grid.origin) + 0.5 * np.array(wk.grid.h)   # a voxel's centre
    ref = direct.forward(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, wk.rho, wk.obs, wk.G)
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):
        with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, dev(wk.obs), mode="direct", precision=prec,
                      max_batch=2, G=wk.G) as plan:
            g, gz = plan.forward(dev(wk.rho), want_gz=True)
            assert rel_l2(g.cpu().numpy(), ref) <= tol
            assert torch.equal(gz, g[..., 2]) and torch.equal(plan.forward(dev(wk.rho)[1])[0], g[1])


@pytest.mark.parametrize("s", [1, 33, 70])
def test_points(s):
    rng = np.random.default_rng(s)
    x, a, rho = rng.uniform(-50, 50, size=(s, 3)), rng.uniform(0.5, 2.0, size=s), rng.normal(2500.0, 300.0, size=s)
    obs = rng.uniform(-70.0, 70.0, size=(50017, 3))
    obs[5] = x[0]
    ref = direct.forward_points(x, a, 1, rho, obs, 1.0)
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):
        with pkg.PointsPlan(dev(x), dev(a), dev(obs), mode="direct", precision=prec, G=1.0) as plan:
            assert rel_l2(plan.forward(dev(rho))[0].cpu().numpy(), ref) <= tol


def test_closed_form():
    wk = wl.random_small(61, n=(2, 1, 1), n_obs=30011, h=(1.0, 1.0, 1.0))
    ref = direct.forward_analytic(wk.grid.n, wk.grid.origin, wk.grid.h, wk.rho, wk.obs, wk.G)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, dev(wk.obs), mode="direct", precision="fp64",
                  voxels="closed_form", G=wk.G) as plan:
        assert rel_l2(plan.forward(dev(wk.rho))[0].cpu().numpy(), ref) <= 1e-12


def median_ms(f):
    for _ in range(3):
        f()
    times = []
    for _ in range(11):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            f()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) / 4)
    return float(np.median(times))


def test_a_million_observers_of_one_voxel():
    obs = dev(np.random.default_rng(1).uniform(0.0, 250.0, size=(1000000, 3)))
    rho = torch.ones((1, 1, 1), device=DEV)
    out = torch.empty_like(obs)
    with pkg.Plan((1, 1, 1), (0.0, 0.0, -250.0), (250.0,) * 3, np.zeros((1, 3)), np.array([8.0]), obs, mode="direct",
                  precision="mixed") as plan:
        took = median_ms(lambda: plan.forward(rho, g=out))
    copy = median_ms(lambda: out.copy_(obs))
    print("%.4f ms, a copy %.4f" % (took, copy))
    assert took <= 4.0 * copy + 0.05
