"""Translations with many columns (four components by several columns per
thread) against the split sums that few columns take: a batch of 64 models in
one plan and the same models one by one.  Both are FP32 sums of at most K
terms per translation, so they agree to a few FP32 roundings; the grid is
ragged (partly empty parents), unaligned to 16-byte rows in one case, and the
degrees include the smallest and the largest."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("n", [(72, 68, 66), (67, 72, 70)])
@pytest.mark.parametrize("p", [1, 2, 5, 10, 15])
def test_many_columns_match_few(p, n):
    wk = wl.random_small(90 + p, n=n, n_obs=400, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, -66.0))
    gen = torch.Generator(device=DEV).manual_seed(p)
    rho = torch.randn((64,) + wk.grid.shape_zyx, generator=gen, device=DEV)
    obs = torch.tensor(wk.obs, dtype=torch.float64, device=DEV)
    args = (wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs)
    with pkg.Plan(*args, precision="mixed", p=p, max_batch=64, G=1.0) as many, \
            pkg.Plan(*args, precision="mixed", p=p, max_batch=1, G=1.0) as few:
        g, _ = many.forward(rho)
        for b in (0, 1, 63):
            ref, _ = few.forward(rho[b])
            assert float((g[b] - ref).norm() / ref.norm()) <= 2e-6
        many.check()
        r = torch.randn((16, wk.n_obs), generator=gen, device=DEV, dtype=torch.float64)
        grad = many.adjoint(r)
        for b in (0, 15):
            ref = few.adjoint(r[b])
            assert float((grad[b] - ref).norm() / ref.norm()) <= 2e-6
        r = torch.randn((16, wk.n_obs, 3), generator=gen, device=DEV, dtype=torch.float64)
        grad = many.adjoint(r, ncomp=3)
        for b in (0, 15):
            ref = few.adjoint(r[b], ncomp=3)
            assert float((grad[b] - ref).norm() / ref.norm()) <= 2e-6
