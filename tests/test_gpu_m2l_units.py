"""The tensor-core M2L at both ways of dealing out its work (units of a tile's
offsets over the grid, or one tile per block), at every number of input chunks
per offset, with source parts that leave tiles empty, and run to run.  Bars:
2e-6 against the SIMT M2L and between the two ways (both carry FP32 rounding
only); repeated runs are bit-identical."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("p", [4, 6, 8, 11, 14, 15])
@pytest.mark.parametrize("n,m", [((9, 17, 12), 40), ((44, 40, 41), 6000)])
def test_chunks_and_parts(n, m, p):
    wk = wl.random_small(300 + p, n=n, n_obs=m, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=1.0)
    obs = torch.tensor(wk.obs, device=DEV)
    rho = torch.tensor(wk.rho, dtype=torch.float32, device=DEV)
    kw = dict(mode="fmm", precision="mixed", p=p, G=1.0)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, m2l="simt", **kw) as plan:
        ref = plan.forward(rho)[0].cpu().numpy()
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, **kw) as plan:
        g = plan.forward(rho)[0].cpu().numpy()
        assert np.array_equal(g, plan.forward(rho)[0].cpu().numpy())
        assert rel_l2(g, ref) <= 2e-6
        total = np.zeros_like(g)
        for part in range(3):
            plan.set_source_part(part, 3)
            total += plan.forward(rho)[0].cpu().numpy()
        assert rel_l2(total, ref) <= 2e-6


def test_more_tiles_than_dealt_out():
    """16 grids at once on 25^3 leaf boxes: 1,960 leaf tiles, one per block;
    one grid: 128 leaf tiles, dealt out."""
    n = (100, 100, 100)
    wk = wl.random_small(320, n=n, n_obs=8, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, 0.0), obs_pad=0.0)
    c = np.arange(25) * 4.0 + 2.3
    obs = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    rho = torch.tensor(np.random.default_rng(5).normal(size=(16,) + n[::-1]), dtype=torch.float32, device=DEV)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, torch.tensor(obs, device=DEV), mode="fmm",
                  precision="mixed", p=7, G=1.0, max_batch=16) as plan:
        all16 = plan.forward(rho)[0].cpu().numpy().reshape(16, -1)
        for b in (0, 15):
            one = plan.forward(rho[b])[0].cpu().numpy().reshape(-1)
            assert rel_l2(all16[b], one) <= 2e-6
