"""The transposed M2M of all children of a parent at once (FP64: the top level of
mixed plans, every level of FP64 ones): the adjoint is the forward's transpose, so
<r, A x> = <A^T r, x> whatever the truncation, to rounding (1e-12 of the product of
norms in FP64, 1e-5 in mixed precision).  Batches on both sides of the two-column
choice, ragged grids whose parents lack children, one and several levels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("precision,p", [("fp64", 9), ("fp64", 14), ("fp64", 16), ("mixed", 11)])
@pytest.mark.parametrize("n,batch", [((33, 29, 31), 1), ((70, 9, 41), 1), ((34, 37, 33), 7)])
def test_transpose(n, batch, precision, p):
    wk = wl.random_small(700 + p, n=n, n_obs=150, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=3.0)
    rng = np.random.default_rng(p)
    r = rng.normal(size=(batch, 150))
    x = rng.normal(size=(batch,) + tuple(n)[::-1])
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, torch.tensor(wk.obs, device=DEV), mode="fmm",
                  precision=precision, p=p, G=1.0, max_batch=batch) as plan:
        g = plan.forward(torch.tensor(x if batch > 1 else x[0], device=DEV))[0].cpu().numpy().reshape(batch, 150, 3)
        grad = plan.adjoint(torch.tensor(r if batch > 1 else r[0], device=DEV)).cpu().numpy().reshape(batch, -1)
    for b in range(batch):
        gz = g[b, :, 2]
        lhs, rhs = float(r[b] @ gz), float(grad[b] @ x[b].ravel())
        err = abs(lhs - rhs) / (np.linalg.norm(r[b]) * np.linalg.norm(gz))
        print("%s p %d batch %d: %.2e" % (precision, p, b, err))
        assert err <= (1e-12 if precision == "fp64" else 1e-5)
