"""The second FP64 stencil of a 2D level is held by hierarchies that have made a
mixed load step, on the levels that the mixed mode takes in FP64, and by no
others."""
import ctypes as C

import pytest

import pfinputs as PI
from tests.gpu_common import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,nc,levels,galerkin,small", [
    (2, (29, 29), 3, 0, [1, 1, 1]),      # 113 x 113 finest
    (2, (30, 29), 3, 0, [1, 1, 0]),      # 117 x 113 finest
    (2, (29, 29), 3, 1, [0, 0, 1]),
    (3, (5, 5, 5), 2, 0, [0, 0]),
])
def test_stencils_held(dim, nc, levels, galerkin, small):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    from tests import native_probe as probe
    lib = probe.load()
    H = pf.mesh_hierarchy_create(dim, nc, levels, 1.0 / (nc[0] - 1), E=1.0, nu=0.25, Gc=1.0)
    pf.pressure_set(H, 1e-3)
    held = lambda: [lib.probe_small_stencil(H.handle, C.c_int(l)) for l in range(levels)]
    x = torch.zeros(H.ndof(), dtype=torch.float64, device="cuda")
    rows = PI.centred_crack_2d() if dim == 2 else PI.disc_network_3d(PI.SEED_3D_PLAIN, 2)
    pf.fractures_set(H, pf.PF_LINE2D if dim == 2 else pf.PF_DISC3D, rows, H.levels[-1][1], x)
    kw = dict(max_cycles=1, coarse_its=1, coarse_model=pf.PF_GALERKIN if galerkin else pf.PF_FIRST_ORDER)
    pf.rmtr_load_step(H, x, pf.default_params(**kw), check=False)
    assert held() == [0] * levels
    pf.rmtr_load_step(H, x, pf.default_params(precision=pf.PF_FP32, **kw), check=False)
    assert held() == small
    H.close()
