"""Rules that are not their own mirror image under 4^3-voxel leaves, mixed precision:
the expansions of the voxel centres, shifted by the rule's nodes.  Against the FP64
oracle (1e-5), at few and at many columns, for one node off the centre and for
several; and the forward takes no more than 1.5 times the centred rule's at 232^3 (with
a P2M of every leaf it took twice that)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from oracle import direct  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"
RULES = {
    "one off centre": ([[0.1, 0.0, 0.0]], [8.0]),
    "one in a corner": ([[-0.9, 0.95, 0.9]], [1.0]),
    "two": ([[0.3, 0.1, -0.2], [-0.5, 0.2, 0.1]], [3.0, 5.0]),
    "five": ([[0.9, 0.1, -0.7], [-0.5, 0.2, 0.1], [0.0, 0.0, 0.0], [0.4, -0.8, 0.3], [-0.1, -0.2, 0.9]],
             [1.0, 2.0, 0.5, 1.5, 3.0]),
}


@pytest.mark.parametrize("name", list(RULES))
@pytest.mark.parametrize("n,batch,p,m", [((29, 22, 17), 1, 12, 500), ((29, 22, 17), 3, 15, 500),
                                         ((176, 172, 24), 4, 11, 4000)])
def test_against_the_oracle(n, batch, p, m, name):
    xi, w = (np.array(v) for v in RULES[name])
    wk = wl.random_small(900 + p, n=n, n_obs=m, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=1.0, B=batch)
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, xi, w, torch.tensor(wk.obs, device=DEV), mode="fmm",
                  precision="mixed", p=p, G=1.0, leaf_vox=4, max_batch=batch) as plan:
        g = plan.forward(torch.tensor(wk.rho, dtype=torch.float32, device=DEV))[0].cpu().numpy().reshape(batch, m, 3)
        assert plan.info.leaf_vox == 4
        plan.check()
    some = np.arange(0, m, max(1, m // 60))
    for b in {0, batch - 1}:
        rho = wk.rho.reshape((batch,) + n[::-1])[b].astype(np.float32).astype(np.float64)
        ref = direct.forward(wk.grid.n, wk.grid.origin, wk.grid.h, xi, w, rho, wk.obs[some], 1.0)
        err = float(np.linalg.norm(g[b][some] - ref) / np.linalg.norm(ref))
        print("%.2e" % err)
        assert err <= 1e-5


def test_not_much_slower_than_the_centre():
    n, s, h = 232, 512, 250.0
    c = (np.arange(s) + 0.5) * (n * h / s)
    obs = torch.tensor(np.stack(np.meshgrid(c, c, [100.0], indexing="ij"), -1).reshape(-1, 3), device=DEV)
    rho = torch.randn((n, n, n), device=DEV)
    ms = []
    for xi in ([[0.0, 0.0, 0.0]], [[0.1, 0.0, 0.0]]):
        with pkg.Plan((n, n, n), (0.0, 0.0, -n * h), (h, h, h), np.array(xi), np.array([8.0]), obs, mode="fmm",
                      precision="mixed", p=10) as plan:
            t = []
            for _ in range(15):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                plan.forward(rho)
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            ms.append(float(np.median(t[4:])))
    print("%.3f ms centred, %.3f ms off centre" % tuple(ms))
    assert ms[1] <= 1.5 * ms[0]
