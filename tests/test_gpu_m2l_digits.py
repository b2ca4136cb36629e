"""The FP64 M2L on the tensor cores (BF16 digits) against the FP64 M2L on the
SIMT cores: degrees with one to five column groups, batches, source parts,
densities over sixteen decades, many and few targets to a tile, more tiles than
are dealt out.  Both carry a few units of 2^-53 of the largest terms; the bar,
1e-13 of the field, leaves a factor of a hundred for cancellation in it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"
BAR = 1e-13


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def fields(wk, obs, rho, m2l, p, batch=1, parts=0):
    with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, torch.tensor(obs, device=DEV), mode="fmm",
                  precision="fp64", p=p, G=1.0, m2l=m2l, max_batch=batch) as plan:
        r = torch.tensor(rho, device=DEV)
        g = plan.forward(r)[0].cpu().numpy()
        assert np.array_equal(g, plan.forward(r)[0].cpu().numpy())
        out = [g]
        for part in range(parts):
            plan.set_source_part(part, parts)
            out.append(plan.forward(r)[0].cpu().numpy())
        plan.check()
    return out


@pytest.mark.parametrize("p", [6, 8, 10, 12, 14, 16])
def test_degrees_and_parts(p):
    wk = wl.random_small(600 + p, n=(44, 40, 41), n_obs=6000, h=(1.0, 1.0, 1.0), origin=(-3.0, 2.0, -30.0), obs_pad=1.0)
    a, b = (fields(wk, wk.obs, wk.rho, m, p, parts=3) for m in ("auto", "simt"))
    if p >= 10:   # the digits are what runs (below it may be the SIMT M2L)
        assert not np.array_equal(a[0], b[0])
    for x, y in zip(a, b):
        print("p %d: %.2e" % (p, rel_l2(x, y)))
        assert rel_l2(x, y) <= BAR


def test_dynamic_range():
    """Blocks of density 1e-8 to 1e8; compared block of observers by block, so
    that the small ones count."""
    n = (48, 48, 48)
    wk = wl.random_small(640, n=n, n_obs=8, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, 0.0), obs_pad=0.0)
    rng = np.random.default_rng(3)
    scale = 10.0 ** rng.integers(-8, 9, size=(6, 6, 6))
    rho = rng.normal(size=n) * np.kron(scale, np.ones((8, 8, 8)))
    c = np.arange(24) * 2.0 + 0.9
    obs = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    a, b = (fields(wk, obs, rho, m, 12)[0] for m in ("auto", "simt"))
    assert not np.array_equal(a, b)
    print("range: %.2e, worst observer %.2e" % (rel_l2(a, b), np.max(np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1))))
    assert rel_l2(a, b) <= BAR
    assert np.max(np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)) <= 1e-11


@pytest.mark.parametrize("batch", [3, 16])
def test_batches(batch):
    n = (36, 33, 30)
    wk = wl.random_small(650, n=n, n_obs=4000, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, -30.0), obs_pad=0.5)
    rho = np.random.default_rng(8).normal(size=(batch,) + n[::-1])
    a, b = (fields(wk, wk.obs, rho, m, 10, batch=batch)[0] for m in ("auto", "simt"))
    assert not np.array_equal(a, b)
    for x, y in zip(a, b):
        assert rel_l2(x, y) <= BAR
    one = fields(wk, wk.obs, rho[1], "auto", 10, batch=batch)[0]
    assert np.array_equal(one, a[1])


def test_more_tiles_than_dealt_out():
    n = (92, 92, 92)
    wk = wl.random_small(660, n=n, n_obs=8, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, 0.0), obs_pad=0.0)
    c = np.arange(46) * 2.0 + 0.9   # eight to a leaf: the plan's size leaves room for the split inputs
    obs = np.stack(np.meshgrid(c, c, c[::2], indexing="ij"), -1).reshape(-1, 3)
    rho = np.random.default_rng(5).normal(size=(16,) + n[::-1])
    a, b = (fields(wk, obs, rho, m, 8, batch=16)[0] for m in ("auto", "simt"))
    assert not np.array_equal(a, b)
    for x, y in zip(a, b):
        assert rel_l2(x, y) <= BAR
