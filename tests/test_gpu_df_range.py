"""The double-float passes over the magnitudes their split of a double has to
handle (exact zeros, values whose lower part leaves FP32's normal range, and
the usual ones), against the library's FP64 gradient and energy: 1e-11 and
1e-12 relative, the parity suite's bounds, down to where FP32's exponent range
ends, and no worse than FP32 itself below."""
import numpy as np
import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(9, 7, 6), (33, 20)])
@pytest.mark.parametrize("scale,tol", [(1.0, 1e-11), (1e-6, 1e-11), (1e-15, 1e-11), (1e-30, 1e-6)])
def test_gradient_df_over_magnitudes(n, scale, tol):
    require_cuda()
    import paper_2007_12908_gb300 as pf
    dim = len(n)
    H, _ = pair(dim, n, 1, 1.0 / (max(n) - 1), p=0.0)
    N = H.nodes()
    x = PI.random_state(5, dim, N, u_scale=1e-3, c_hi=0.9) * scale
    x[::7] = 0.0
    x[1::11] = -0.0
    xd = dev(x)
    # at p = 0 and small c the c rows are linear in the state: relative to it
    g, gd = host(pf.gradient(H, 0, xd)), host(pf.gradient_df(H, 0, xd))
    assert relinf(gd[dim * N:], g[dim * N:]) <= tol
    if scale >= 1e-15:
        assert relinf(gd, g) <= tol
    if scale == 1.0:
        e = pf.energy(H, 0, xd)
        assert abs(pf.energy_df(H, 0, xd) - e) <= 1e-12 * abs(e)
    H.close()
