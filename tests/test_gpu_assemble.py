"""The FP64 stencil assembly at the sizes where its node tiles (8 x 4 nodes in
3D, 32 in 2D) and its chunks of layers end: every block of the stencil enters
the product with a random vector, which is compared with the oracle's
matrix-free product within the FP64 parity tolerance of the suite (1e-10,
relative, max-norm), and the operator is symmetric to FP64 rounding."""
import numpy as np
import pytest

import pfinputs as PI
from oracle import pf_oracle as O
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2, 2), (3, 2), (32, 3), (33, 40), (65, 2), (31, 130),
                               (2, 2, 2), (8, 4, 2), (9, 5, 3), (7, 3, 20), (16, 8, 5), (17, 13, 4), (2, 9, 33)])
def test_assembled_hessian_matches_oracle(n):
    require_cuda()
    import paper_2007_12908_gb300 as pf
    dim = len(n)
    H, Ho = pair(dim, n, 1, 1.0 / (max(n) - 1), nu=0.25, p=5e-3)
    g = Ho.fine
    x = PI.random_state(21, dim, g.N, u_scale=1e-3, c_hi=1.0)
    pf.hessvec_lag_set(H, 0, dev(x))
    vs = [PI.random_direction(22 + k, x.size) for k in range(2)]
    got = [host(pf.hessvec_lagged(H, 0, dev(v))) for v in vs]
    for v, y in zip(vs, got):
        assert relinf(y, O.hessvec(g, Ho.prm, x, v)) <= 1e-10
    a, b = float(np.dot(vs[0], got[1])), float(np.dot(vs[1], got[0]))
    assert abs(a - b) <= 1e-13 * np.linalg.norm(vs[0]) * np.linalg.norm(got[1])
    # a second lag replaces every entry (none is left from the first)
    x2 = PI.random_state(31, dim, g.N, u_scale=1e-3, c_hi=1.0)
    pf.hessvec_lag_set(H, 0, dev(x2))
    assert relinf(host(pf.hessvec_lagged(H, 0, dev(vs[0]))), O.hessvec(g, Ho.prm, x2, vs[0])) <= 1e-10
    H.close()


@pytest.mark.parametrize("nc,L", [((34, 3), 2), ((17, 3), 3), ((2, 2), 5), ((2, 17, 3), 2), ((9, 5, 2), 2),
                                  ((2, 2, 2), 4), ((3, 2, 5), 3)])
def test_galerkin_stencils_at_tile_edges(nc, L):
    """The moment form of the Galerkin operators where its CTAs of 32 coarse
    elements and the assembly's tiles end, and over up to four re-expansions:
    R H I of the oracle within FP32 rounding (2e-5 as in the parity suite)."""
    import torch
    require_cuda()
    import paper_2007_12908_gb300 as pf
    dim = len(nc)
    H, Ho = pair(dim, nc, L, 1.0 / (max(nc) - 1), nu=0.25, p=3e-2, k_res=1e-3)
    x32 = PI.random_state(71, dim, Ho.fine.N, u_scale=0.05, c_hi=0.9).astype(np.float32)
    pf.galerkin_set(H, dev(x32))
    x = x32.astype(np.float64)
    for l in range(L - 1):
        v = PI.random_direction(72 + l, Ho.ndof(l)).astype(np.float32).astype(np.float64)
        w = v
        for k in range(l, L - 1):
            w = Ho.transfers[k].prolong(w)
        w = O.hessvec(Ho.fine, Ho.prm, x, w)
        for k in reversed(range(l, L - 1)):
            w = Ho.transfers[k].restrict(w)
        assert relinf(host(pf.galerkin_apply(H, l, dev(v, torch.float32))), w) <= 2e-5
        assert relinf(host(pf.galerkin_apply(H, l, dev(v))), w) <= 2e-5
    H.close()
