"""The FP64 M2L by BF16 digits with more (tile, column group) pairs than it deals
out (1,792): one pair to a block, no partial rows.  Against the FP64 M2L on the SIMT
cores, at its bar (1e-13 of the field), forward and from a part of the sources."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"
BAR = 1e-13
DEALT_OUT = 1792   # pairs, at most, that are dealt out over the SMs


def test_a_pair_to_a_block():
    n, p = (192, 192, 192), 8
    c = np.arange(96) * 2.0 + 0.9   # eight observers to each of 48^3 leaves
    obs = torch.tensor(np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3), device=DEV)
    rho = torch.tensor(np.random.default_rng(5).normal(size=n), device=DEV)
    xi, w = wl.gauss_rule(1)
    out = []
    for m2l in ("auto", "simt"):
        with pkg.Plan(n, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), xi, w, obs, mode="fmm", precision="fp64", p=p, G=1.0,
                      m2l=m2l) as plan:
            # tiles of 128 boxes of a level and parity class, column groups of up to 64 components
            tiles = sum(-(-plan.info.n_target_boxes[level] // 128) for level in range(2, plan.info.L + 1))
            assert tiles * -(-(p + 1) ** 2 // 64) > DEALT_OUT
            whole = plan.forward(rho)[0].cpu().numpy()
            plan.set_source_part(1, 3)
            out.append((whole, plan.forward(rho)[0].cpu().numpy()))
            plan.check()
    for a, b in zip(*out):
        assert not np.array_equal(a, b)   # the digits are what ran
        err = float(np.linalg.norm(a - b) / np.linalg.norm(b))
        print("%.2e" % err)
        assert err <= BAR
