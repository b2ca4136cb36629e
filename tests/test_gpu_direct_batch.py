"""A batch member's direct sums are the same bits alone and in any batch: voxels in
both precisions, closed-form voxels and points, at observer counts where a batch's
tiles together would ask for another split of the sources than one member's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"
BATCH = 3


def dev(a, dtype=torch.float64):
    return torch.tensor(a, dtype=dtype, device=DEV)


def check(plan, rho):
    all3 = plan.forward(rho)[0]
    for b in range(BATCH):
        assert torch.equal(plan.forward(rho[b].contiguous())[0], all3[b]), b


@pytest.mark.parametrize("precision,voxels,n,m", [("fp64", "quadrature", (31, 20, 9), 2560), ("fp64", "quadrature", (31, 20, 9), 20),
                                                  ("mixed", "quadrature", (31, 20, 9), 2560),
                                                  ("fp64", "closed_form", (9, 8, 5), 1300)])
def test_voxels(precision, voxels, n, m):
    wk = wl.random_small(80 + m, n=n, n_obs=m, B=BATCH, h=(1.0, 1.0, 1.0))
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, dev(wk.obs), mode="direct", precision=precision,
                  max_batch=BATCH, G=1.0, voxels=voxels) as plan:
        check(plan, dev(wk.rho))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_points(precision):
    rng = np.random.default_rng(90)
    x, obs = rng.uniform(-50.0, 50.0, size=(6000, 3)), rng.uniform(-70.0, 70.0, size=(2560, 3))
    with pkg.PointsPlan(dev(x), dev(rng.uniform(0.5, 2.0, size=6000)), dev(obs), mode="direct", precision=precision,
                        max_batch=BATCH, G=1.0) as plan:
        check(plan, dev(rng.normal(2500.0, 300.0, size=(BATCH, 6000))))
