"""The SIMT M2L (columns folded by mirror symmetry) at every number of columns
per block it chooses from, for degrees up to the largest, with observers
inside, around and on one side of the sources, against the FP64 oracle; and
the FP32 form against the tensor cores.  Bars: the FMM's own (1e-6 at p >= 14
in FP64, 1e-5 in mixed precision)."""
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


# (grid, observers, pad): few boxes; a plane's worth; a filled volume
CASES = [((9, 17, 12), 40, 2.0), ((36, 33, 30), 900, 1.0), ((44, 40, 41), 6000, 0.0)]


@pytest.mark.parametrize("p", [14, 16])
@pytest.mark.parametrize("n,m,pad", CASES)
def test_fp64_columns_per_block(n, m, pad, p):
    wk = wl.random_small(120 + p, n=n, n_obs=m, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=pad)
    ref = direct.forward(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, wk.rho, wk.obs, wk.G)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, torch.tensor(wk.obs, device=DEV), mode="fmm",
                  precision="fp64", p=p, G=1.0) as plan:
        g = plan.forward(torch.tensor(wk.rho, device=DEV))[0].cpu().numpy()
        assert rel_l2(g, ref) <= 1e-6
        r = np.random.default_rng(p).normal(size=m)
        grad = plan.adjoint(torch.tensor(r, device=DEV)).cpu().numpy()
    vox = np.arange(0, wk.rho.size, 97)
    aref = direct.adjoint_subset(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, wk.obs, r, wk.G, vox)
    assert rel_l2(grad.ravel()[vox], np.asarray(aref).ravel()) <= 1e-6


@pytest.mark.parametrize("n,m,pad", CASES)
def test_fp32_simt_matches_tensor_cores(n, m, pad):
    wk = wl.random_small(140, n=n, n_obs=m, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=pad)
    obs = torch.tensor(wk.obs, device=DEV)
    rho = torch.tensor(wk.rho, dtype=torch.float32, device=DEV)
    out = []
    for m2l in ("simt", "auto"):
        with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, mode="fmm", precision="mixed", p=12,
                      G=1.0, m2l=m2l) as plan:
            out.append(plan.forward(rho)[0].cpu().numpy())
    assert rel_l2(out[0], out[1]) <= 2e-6
