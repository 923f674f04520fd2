"""The trust-region subproblem of a small level in one launch, at the edges of
its split (a warp, a CTA and the device of rows, and the first grid beyond it),
with and without the preconditioner, with budgets that end in the middle of a
CG run: one cycle of a one-level load step against the oracle's, which takes
the same decisions."""
import numpy as np
import pytest

import pfinputs as PI
from oracle import pf_oracle as O
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu

# FP64 throughout, the sums in another order: some 1e-13 per iteration, grown
# by the conditioning over at most 24 iterations
TOL = 1e-9


@pytest.mark.parametrize("dim,n,cg,restarts,pre", [
    (2, (3, 3), 12, 100, 1),           # less than a warp of rows
    (2, (40, 40), 12, 100, 1),         # 4800 rows: 32 to a CTA
    (2, (41, 40), 5, 100, 0),          # 4920 rows: 64 to a CTA
    (2, (113, 114), 12, 0, 1),         # 38646 rows: 128 to a CTA, the last ragged
    (2, (115, 113), 12, 0, 1),         # 38985 rows: separate launches
    (3, (5, 4, 3), 12, 100, 1),
    (3, (32, 19, 16), 8, 100, 0),      # 38912 rows: the most
    (3, (23, 21, 20), 8, 100, 1),      # 38640 rows
])
def test_one_cycle_matches_oracle(dim, n, cg, restarts, pre):
    require_cuda()
    import paper_2007_12908_gb300 as pf
    h = 1.0 / (max(n) - 1)
    H, Ho = pair(dim, n, 1, h, nu=0.3 if dim == 2 else 0.25, p=1e-2)
    N = Ho.fine.N
    xo = np.zeros((dim + 1) * N)
    xo[dim * N:] = np.random.default_rng(5).uniform(0.0, 0.9, N) ** 4
    x = dev(xo)
    kw = dict(coarse_its=2, cg_coarse=cg, max_restarts=restarts, max_cycles=1, rtol=1e-13)
    ro = O.rmtr_load_step(Ho, xo, O.TRParams(precondition=bool(pre), **kw), p=1e-2)
    st = pf.rmtr_load_step(H, x, pf.default_params(precondition=pre, **kw), check=False)
    assert st["cg"] == ro.stats["cg"]
    assert relinf(host(x), ro.x) <= TOL


@pytest.mark.parametrize("nc", [(57, 57), (58, 57)])
def test_mixed_2d_with_small_levels(nc):
    """Mixed 2D load steps whose levels are all small (113 x 113), and whose
    finest is not (115 x 113), against the FP64 step."""
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(2, nc, 2, 1 / 56, p=1e-3)
    x = torch.zeros(H.ndof(), dtype=torch.float64, device="cuda")
    pf.fractures_set(H, pf.PF_LINE2D, PI.centred_crack_2d(), Ho.fine.h, x)
    x64 = x.clone()
    s64 = pf.rmtr_load_step(H, x64, pf.default_params(rtol=1e-12))
    s32 = pf.rmtr_load_step(H, x, pf.default_params(rtol=1e-12, precision=pf.PF_FP32))
    assert s64["converged"] == 1 and s32["converged"] == 1
    assert abs(s32["energy"] - s64["energy"]) <= 1e-8 * abs(s64["energy"])
