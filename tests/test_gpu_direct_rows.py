"""The axis along which a direct sum's rows run: long rows are fewer work units to share
out, so few stations over a grid whose x side is the short one must not wait for them.
6 x 12 x 29 voxels against 15 x 12 x 12, 3% more of them with rows along x: 1.6 leaves
room for the shorter pieces (1.1 to 1.3 by count) and the timing's spread; rows along z
took 2.2 times as long.  Both against the FP64 oracle at the direct sums' bar."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def sum_us(n):
    wk = wl.random_small(7, n=n, npts=1, n_obs=227, B=2)
    ref = direct.forward(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, wk.rho, wk.obs, wk.G)
    obs, rho = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (wk.obs, wk.rho))
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, obs, mode="direct", precision="fp64", max_batch=2,
                  G=wk.G) as plan:
        g = plan.forward(rho)[0].cpu().numpy()
        assert np.linalg.norm(g - ref) <= 1e-12 * np.linalg.norm(ref)
        times = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                plan.forward(rho)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 50.0)
    return float(np.median(times))


def test_few_stations_short_x():
    short, cube = sum_us((6, 12, 29)), sum_us((15, 12, 12))
    print("%.1f us, %.1f" % (short, cube))
    assert short <= 1.6 * cube
