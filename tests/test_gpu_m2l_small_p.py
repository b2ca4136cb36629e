"""The FP32 SIMT M2L at the degrees whose blocks have fewer threads than source
rows to look up (p = 1, 2, 3), with enough columns for eight to a block: forward
and transpose against the FP64 SIMT M2L of the same degree and against the tensor
cores.  Bars: the mixed precision's 1e-5, and the 2e-6 between its two M2Ls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1107_5951_gb300 as pkg  # noqa: E402
from paper_1107_5951_gb300 import workloads as wl  # noqa: E402

DEV = "cuda:0"


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("p", [1, 2, 3])
def test_fp32_simt_small_degrees(p):
    n = (64, 64, 64)
    wk = wl.random_small(700 + p, n=n, n_obs=8, h=(1.0, 1.0, 1.0), origin=(0.0, 0.0, 0.0), obs_pad=0.0)
    c = np.arange(16) * 4.0 + 2.3   # an observer in each of the 4,096 leaves
    obs = np.stack(np.meshgrid(c, c, c, indexing="ij"), -1).reshape(-1, 3)
    rho = np.random.default_rng(p).normal(2500.0, 300.0, size=n)
    r = np.random.default_rng(30 + p).normal(size=(len(obs), 3))
    out = []
    for precision, m2l, dtype in (("mixed", "simt", torch.float32), ("fp64", "simt", torch.float64),
                                  ("mixed", "auto", torch.float32)):
        with pkg.Plan(wk.grid.n, wk.grid.origin, wk.grid.h, wk.xi, wk.w, torch.tensor(obs, device=DEV), mode="fmm",
                      precision=precision, p=p, G=1.0, m2l=m2l) as plan:
            boxes = sum(plan.info.n_target_boxes[level] for level in range(2, plan.info.L + 1))
            assert boxes >= 16 * torch.cuda.get_device_properties(0).multi_processor_count
            g = plan.forward(torch.tensor(rho, dtype=dtype, device=DEV))[0].cpu().numpy()
            grad = plan.adjoint(torch.tensor(r, device=DEV), ncomp=3).cpu().numpy()
            plan.check()
        out.append((g, grad))
    for a, ref, tensor in zip(*out):
        print("p %d: %.2e %.2e" % (p, rel_l2(a, ref), rel_l2(a, tensor)))
        assert rel_l2(a, ref) <= 1e-5
        assert rel_l2(a, tensor) <= 2e-6
