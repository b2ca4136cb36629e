"""The FP64 near field beside the digit M2L takes as much shared memory as spreads its
blocks over the SMs: grids whose blocks fill one to six SM places each, among them the
three to an SM that need between 31 and 47 KB beside 17 KB of static memory (a launch
without the opt-in was refused).  Against the mixed plan of the same degree, which has
the same truncation: its field is within 1e-5 of the largest, the bound leaves ten times
that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("leaves", [8, 11, 13, 15, 16, 18, 20])
def test_blocks_per_sm(leaves):
    n, h = 4 * leaves, 250.0
    c = (np.arange(2 * n) + 0.5) * (h / 2)
    obs = torch.tensor(np.stack(np.meshgrid(c, c, [0.0], indexing="ij"), -1).reshape(-1, 3), device=DEV)
    xi, w = wl.gauss_rule(1)
    rho = torch.tensor(np.random.default_rng(3).normal(0.0, 150.0, size=(n, n, n)), device=DEV)
    g = {}
    for precision in ("mixed", "fp64"):
        with pkg.Plan((n, n, n), (0.0, 0.0, -n * h), (h, h, h), xi, w, obs, mode="fmm", precision=precision, p=10) as plan:
            g[precision] = plan.forward(rho)[0].cpu().numpy()
    assert np.abs(g["fp64"] - g["mixed"]).max() <= 1e-4 * np.abs(g["mixed"]).max()
