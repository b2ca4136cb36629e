"""The offsets a tensor-core M2L tile runs, found from the window's extent alone
(every source counts) against testing each offset (source parts), on windows
thinner than an interaction list on one, two and all axes.  Bar: the two ways
and the SIMT M2L differ by FP32 rounding only, 2e-6; an offset left out would
drop a whole source box."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", [(3, 90, 61), (64, 5, 3), (33, 33, 2), (17, 18, 19), (1, 1, 130)])
def test_thin_windows(n):
    wk = wl.random_small(340, n=n, n_obs=20000, h=(1.0, 1.0, 1.0), origin=(5.0, -3.0, -20.0), obs_pad=0.5)
    obs = torch.tensor(wk.obs, device=DEV)
    rho = torch.tensor(wk.rho, dtype=torch.float32, device=DEV)
    kw = dict(mode="fmm", precision="mixed", p=8, G=1.0)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, m2l="simt", **kw) as plan:
        ref = plan.forward(rho)[0].cpu().numpy()
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, **kw) as plan:
        g = plan.forward(rho)[0].cpu().numpy()
        total = np.zeros_like(g)
        for part in range(2):
            plan.set_source_part(part, 2)
            total += plan.forward(rho)[0].cpu().numpy()
    assert rel_l2(g, ref) <= 2e-6
    assert rel_l2(g, total) <= 2e-6
