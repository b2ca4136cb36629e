"""Device memory of plans: a 32^3 grid under a plane of 256^2 stations stays within
20 MB in mixed precision (the M2L's partial rows take what the targets need, not
whole tiles for every SM), and a server whose budget holds such a request's
expansions, buffers and scratch (20 MB; FP64 25 MB) takes it, with the same field
to rounding; so does one whose budget is some MB short of a small grid's with
observers throughout, which then deals its M2L out to fewer blocks, or not at all."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("precision,p,dtype,budget,bar", [("mixed", 12, np.float32, 20e6, 2e-6),
                                                          ("fp64", 14, np.float64, 25e6, 1e-13)])
def test_small_request_fits(precision, p, dtype, budget, bar):
    n, h = 32, 250.0
    xi, w = wl.gauss_rule(1)
    c = (np.arange(256) + 0.5) * (n * h / 256)
    obs = np.stack(np.meshgrid(c, c, [0.0], indexing="ij"), -1).reshape(-1, 3)
    rho = np.random.default_rng(4).normal(0.0, 150.0, size=(n, n, n)).astype(dtype)
    geo = ((n, n, n), (0.0, 0.0, -n * h), (h, h, h), xi, w)
    with pkg.Plan(*geo, torch.tensor(obs, device=DEV), mode="fmm", precision=precision, p=p) as plan:
        want = plan.forward(torch.tensor(rho, device=DEV))[0].cpu().numpy()
        assert plan.info.device_bytes <= budget
        assert plan.info.device_bytes <= pkg.plan_bytes(*geo, len(obs), mode="fmm", precision=precision, p=p)
    with pkg.Server(slots=1, precision=precision, p=p, mem_budget=int(budget)) as srv:
        srv.register(1, *geo, obs)
        _, g, _ = srv.wait(srv.submit(1, rho, want_g=True))
        assert srv.stats()["resident_bytes"] <= budget
    assert rel_l2(g, want) <= bar


@pytest.mark.parametrize("short", [1e6, 6e6, 9e6])
@pytest.mark.parametrize("precision,p,dtype,bar", [("mixed", 12, np.float32, 2e-6), ("fp64", 10, np.float64, 1e-13)])
def test_short_budget(precision, p, dtype, bar, short):
    wk = wl.random_small(750, n=(44, 40, 41), n_obs=6000, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=1.0)
    geo = (wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w)
    rho = wk.rho.astype(dtype)
    with pkg.Plan(*geo, torch.tensor(wk.obs, device=DEV), mode="fmm", precision=precision, p=p) as plan:
        want = plan.forward(torch.tensor(rho, device=DEV))[0].cpu().numpy()
    need = pkg.plan_bytes(*geo, len(wk.obs), mode="fmm", precision=precision, p=p) + rho.nbytes + 32 * len(wk.obs)
    with pkg.Server(slots=1, precision=precision, p=p, mem_budget=int(need - short)) as srv:
        srv.register(1, *geo, wk.obs)
        _, g, _ = srv.wait(srv.submit(1, rho, want_g=True))
    assert rel_l2(g, want) <= bar
