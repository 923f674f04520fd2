"""The transfer kernels at the sizes where their column tiles and layer chunks
end (32 x 4 coarse columns, chunks of 1 to 8 layers), against the oracle's
sparse transfers: FP64 within a few ulp of the at most 27 terms of a sum, FP32
within the same number of FP32 ulp, the bounds exactly, special values
included."""
import numpy as np
import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, pair, relinf, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [(2, 2), (33, 5), (64, 4), (2, 9), (2, 2, 2), (33, 4, 3), (32, 5, 9),
                                (3, 2, 17), (65, 33, 10)])
def test_transfers_at_tile_and_chunk_edges(nc):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(len(nc), nc, 2, 1.0 / (max(nc) - 1))
    T = Ho.transfers[0]
    for scale, dtype, tol in ((1.0, None, 1e-15), (1.0, torch.float32, 5e-7), (1e300, None, 1e-15)):
        vc = PI.random_direction(11, H.ndof(0), scale)
        vf = PI.random_direction(12, H.ndof(1), scale)
        if dtype is not None:
            vc, vf = vc.astype(np.float32).astype(np.float64), vf.astype(np.float32).astype(np.float64)
        assert relinf(host(pf.prolong(H, 0, dev(vc, dtype))), T.prolong(vc)) <= 2 * tol
        assert relinf(host(pf.restrict(H, 0, dev(vf, dtype))), T.restrict(vf)) <= 2 * tol
        assert relinf(host(pf.project(H, 0, dev(vf, dtype))), T.project(vf)) <= 2 * tol
    # subnormal values halve as IEEE multiplication halves them
    tiny = np.full(H.ndof(0), 5e-324)
    assert np.all(host(pf.prolong(H, 0, dev(tiny))) <= 5e-324)
    H.close()


@pytest.mark.parametrize("nc", [(33, 5), (3, 2, 9)])
def test_coarse_bounds_special_values(nc):
    """Infinities, signed zeros and the largest values, and a NaN, which never
    wins (as with fmax and fmin)."""
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H, Ho = pair(len(nc), nc, 2, 1.0 / (max(nc) - 1))
    n, N = H.ndof(1), H.nodes(1)
    pool = np.array([-np.inf, np.inf, 0.0, -0.0, 1.7e308, -1.7e308, 5e-324, -5e-324, 1.0, -1.0, np.nan, -np.nan])
    lo = pool[PI.rng(5).integers(0, len(pool), n)]
    hi = pool[PI.rng(6).integers(0, len(pool), n)]
    lc, hc = pf.coarse_bounds(H, 0, dev(lo), dev(hi))
    lc, hc = host(lc), host(hc)
    shape = (len(nc) + 1,) + tuple(reversed([2 * (v - 1) + 1 for v in nc]))
    for v, got, op, start in ((lo, lc, np.fmax, -np.inf), (hi, hc, np.fmin, np.inf)):
        t = np.where(np.isnan(v), start, v).reshape(shape)
        for ax in range(1, len(nc) + 1):
            t = np.moveaxis(t, ax, -1)
            out = t[..., 0::2].copy()
            out[..., 1:] = op(out[..., 1:], t[..., 1::2])
            out[..., :-1] = op(out[..., :-1], t[..., 1::2])
            t = np.moveaxis(out, -1, ax)
        assert np.array_equal(got, t.reshape(-1))
    H.close()
