"""The stencil assembly where a CTA marches over several node layers: 4 layers
(FP64, 33 x 25 x 30 nodes) and 3 (FP32, a stored Galerkin level of 33 x 25 x 29),
the last chunk of 2, compared in full with the oracle within the tolerances of the
parity suite.  The grids of the other assembly tests all have one layer to a chunk."""
import numpy as np
import pytest

import pfinputs as PI
from oracle import pf_oracle as O
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu


def test_fp64_hessian():
    require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(3, (33, 25, 30), 1, 1 / 32, nu=0.25, p=5e-3)
    g = Ho.fine
    x = PI.random_state(21, 3, g.N, u_scale=1e-3, c_hi=1.0)
    pf.hessvec_lag_set(H, 0, dev(x))
    for k in range(2):
        v = PI.random_direction(22 + k, x.size)
        assert relinf(host(pf.hessvec_lagged(H, 0, dev(v))), O.hessvec(g, Ho.prm, x, v)) <= 1e-10
    H.close()


def test_fp32_galerkin():
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(3, (33, 25, 29), 2, 1 / 32, nu=0.25, p=3e-2, k_res=1e-3)
    x32 = PI.random_state(71, 3, Ho.fine.N, u_scale=0.05, c_hi=0.9).astype(np.float32)
    pf.galerkin_set(H, dev(x32))
    v = PI.random_direction(72, Ho.ndof(0)).astype(np.float32).astype(np.float64)
    T = Ho.transfers[0]
    w = T.restrict(O.hessvec(Ho.fine, Ho.prm, x32.astype(np.float64), T.prolong(v)))
    assert relinf(host(pf.galerkin_apply(H, 0, dev(v, torch.float32))), w) <= 2e-5
    assert relinf(host(pf.galerkin_apply(H, 0, dev(v))), w) <= 2e-5
    H.close()
