"""The first iteration of a CG run takes the direction its start wrote; every
later one takes M^-1 r + beta p, also where r . M^-1 r, and so beta, has become
zero in mid-run."""
import ctypes as C

import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, relinf, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta,later", [(0.0, False), (0.0, True), (1e-60, True), (0.5, True)])
@pytest.mark.parametrize("pre", [True, False])
def test_direction_of_an_iteration(beta, later, pre):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    from tests import native_probe as probe
    lib = probe.load()
    H = pf.mesh_hierarchy_create(3, (17, 10, 12), 1, 1 / 16, E=1.0, nu=0.25, Gc=1.0)
    pf.tile_variant_set(H, 0, 1)  # element-owned tiles
    n = H.ndof()
    x, p, r, m = (dev(PI.random_direction(k, n), torch.float32) for k in (1, 2, 3, 4))
    q = torch.empty_like(p)
    old = p.clone()
    rc = lib.probe_cg_product(H.handle, C.c_int(0), probe.ptr(x), probe.ptr(p), probe.ptr(q), probe.ptr(r),
                              probe.ptr(m if pre else None), C.c_double(beta), C.c_int(7),
                              C.c_int(9 if later else 7))
    assert rc == 0
    want = torch.addcmul(beta * old.double(), m.double(), r.double()) if pre else r.double() + beta * old.double()
    want = want if later else old.double()
    assert relinf(host(p), host(want)) <= (2e-7 if later else 0.0)
    assert relinf(host(q), host(pf.hessvec(H, 0, x, p))) <= 1e-6
    H.close()
