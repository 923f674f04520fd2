"""The transfers where a thread marches over several coarse layers of its column
(chunks of 4 and of 2 layers, from about 1,200 blocks on; the grids of the other
transfer tests are all below, with one layer to a thread), the last chunk ragged,
with NaNs and infinities across a chunk's edge, against the same operations axis
by axis in NumPy: within a few ulp of a sum's at most 27 terms, the bounds
exactly."""
import numpy as np
import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, relinf, require_cuda

pytestmark = pytest.mark.gpu

NC = [(65, 65, 63), (49, 48, 31)]


def _prolong(a):
    for ax in (1, 2, 3):
        a = np.moveaxis(a, ax, -1)
        out = np.empty(a.shape[:-1] + (2 * a.shape[-1] - 1,))
        out[..., 0::2] = a
        out[..., 1::2] = 0.5 * a[..., :-1] + 0.5 * a[..., 1:]
        a = np.moveaxis(out, -1, ax)
    return a


def _gather(a, op, half):
    for ax in (1, 2, 3):
        a = np.moveaxis(a, ax, -1)
        out = a[..., 0::2].copy()
        out[..., 1:] = op(out[..., 1:], half * a[..., 1::2])
        out[..., :-1] = op(out[..., :-1], half * a[..., 1::2])
        a = np.moveaxis(out, -1, ax)
    return a


def _shape(n):
    return (4, n[2], n[1], n[0])


def _marked(v, n, z):
    v = v.reshape(_shape(n)).copy()
    v[0, z, 3, 5] = np.nan
    v[1, z + 1, 2, 7] = np.nan
    v[2, z, 4, 4] = np.inf
    return v


@pytest.mark.parametrize("nc", NC)
def test_transfers(nc):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H = pf.mesh_hierarchy_create(3, nc, 2, 1.0 / (max(nc) - 1))
    nf = [2 * v - 1 for v in nc]
    for dtype, tol in ((torch.float64, 2e-15), (torch.float32, 1e-6)):
        vc = host(dev(PI.random_direction(11, H.ndof(0)), dtype))
        vf = host(dev(PI.random_direction(12, H.ndof(1)), dtype))
        ones = np.ones(_shape(nf))
        for src, fn, ref in ((_marked(vc, nc, 3), pf.prolong, _prolong),
                             (_marked(vf, nf, 7), pf.restrict, lambda a: _gather(a, np.add, 0.5)),
                             (_marked(vf, nf, 7), pf.project,
                              lambda a: _gather(a, np.add, 0.5) / _gather(ones, np.add, 0.5))):
            got = host(fn(H, 0, dev(src.reshape(-1), dtype)))
            want = ref(src).reshape(-1)
            assert np.array_equal(np.isnan(got), np.isnan(want))
            fin = np.isfinite(want)
            assert np.array_equal(got[~fin & ~np.isnan(want)], want[~fin & ~np.isnan(want)])
            assert relinf(got[fin], want[fin]) <= tol
    H.close()


@pytest.mark.parametrize("nc", NC)
def test_bounds(nc):
    require_cuda()
    import paper_2007_12908_gb300 as pf
    H = pf.mesh_hierarchy_create(3, nc, 2, 1.0 / (max(nc) - 1))
    nf = [2 * v - 1 for v in nc]
    pool = np.array([-np.inf, np.inf, 0.0, -0.0, 1.7e308, -1.7e308, 5e-324, -5e-324, 1.0, -1.0, np.nan, -np.nan])
    lo = pool[PI.rng(5).integers(0, len(pool), H.ndof(1))]
    hi = pool[PI.rng(6).integers(0, len(pool), H.ndof(1))]
    lc, hc = pf.coarse_bounds(H, 0, dev(lo), dev(hi))
    for v, got, op, start in ((lo, host(lc), np.fmax, -np.inf), (hi, host(hc), np.fmin, np.inf)):
        want = _gather(np.where(np.isnan(v), start, v).reshape(_shape(nf)), op, 1.0)
        assert np.array_equal(got, want.reshape(-1))
    H.close()
