"""The 3D FP32 Hessian product at the edges of its tiles (element-owned 8^3,
node-owned 8^3 and 4^3): one tile, one element or node more, two layers of
elements, against the oracle."""
import numpy as np
import pytest

import pfinputs as PI
from oracle import pf_oracle as O
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu

# some 30 FP32 roundings on the longest path of a row's largest terms
TOL = 30 * 2.0 ** -24


@pytest.mark.parametrize("n", [(9, 9, 9), (10, 9, 17), (17, 18, 3), (25, 8, 5), (5, 4, 33)])
@pytest.mark.parametrize("variant", [1, 2, 3])
def test_tile_edges(n, variant):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(3, n, 1, 0.125, nu=0.25, p=5e-3)
    g = Ho.fine
    x = PI.random_state(31, 3, g.N, u_scale=1e-3, c_hi=1.0)
    v = PI.random_direction(32, x.size)
    x32, v32 = x.astype(np.float32), v.astype(np.float32)
    pf.tile_variant_set(H, 0, variant)
    ho = O.hessvec(g, Ho.prm, x32.astype(np.float64), v32.astype(np.float64))
    out = pf.hessvec(H, 0, dev(x32), dev(v32))
    assert relinf(host(out), ho) <= TOL
