"""The subproblem of a small level when its one launch is not to be had: separate
launches do the same arithmetic (FP64 in the mixed mode's small 2D levels too),
and a grid barrier whose wait runs out leaves a load step that equals one by
separate launches from its start, bit for bit, and a usable hierarchy."""
import ctypes as C

import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, relinf, require_cuda

pytestmark = pytest.mark.gpu

CASES = [(2, (17, 17), 2, False, 0), (2, (17, 17), 2, True, 0), (2, (17, 17), 2, True, 1), (3, (5, 5, 5), 2, False, 0),
         (3, (5, 5, 5), 2, True, 1)]


def _start(pf, dim, nc, levels):
    torch = require_cuda()
    H = pf.mesh_hierarchy_create(dim, nc, levels, 1.0 / (nc[0] - 1), E=1.0, nu=0.25, Gc=1.0)
    pf.pressure_set(H, 1e-2)
    x = torch.zeros(H.ndof(), dtype=torch.float64, device="cuda")
    x[dim * H.nodes():] = dev(PI.rng(5).uniform(0.0, 0.9, H.nodes()) ** 4)
    return H, x


def _params(pf, mixed, galerkin, **kw):
    if mixed:
        kw["precision"] = pf.PF_FP32
    return pf.default_params(coarse_model=pf.PF_GALERKIN if galerkin else pf.PF_FIRST_ORDER, **kw)


@pytest.mark.parametrize("dim,nc,levels,mixed,galerkin", CASES[:2] + CASES[3:4])
def test_separate_launches_do_the_same_arithmetic(dim, nc, levels, mixed, galerkin):
    """FP64 sums in another order, grown by the conditioning over some 100
    iterations of one cycle: 1e-8; FP32 levels are 6e-8 off."""
    require_cuda()
    import paper_2007_12908_gb300 as pf
    from tests import native_probe as probe
    lib = probe.load()
    out = []
    for separate in (False, True):
        H, x = _start(pf, dim, nc, levels)
        if separate:
            lib.probe_separate_launches(H.handle)
        st = pf.rmtr_load_step(H, x, _params(pf, mixed, galerkin, max_cycles=1, cg_coarse=12, coarse_its=2, rtol=1e-13),
                               check=False)
        out.append((host(x), st["cg"]))
        H.close()
    assert out[0][1] == out[1][1]
    assert relinf(out[1][0], out[0][0]) <= 1e-8


@pytest.mark.parametrize("dim,nc,levels,mixed,galerkin", CASES)
def test_a_wait_that_runs_out(dim, nc, levels, mixed, galerkin):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    from tests import native_probe as probe
    lib = probe.load()
    out = []
    for stuck in (True, False):
        H, x = _start(pf, dim, nc, levels)
        if stuck:
            assert lib.probe_stuck_barrier(H.handle, C.c_longlong(2000)) == 0
        else:
            lib.probe_separate_launches(H.handle)
        runs = []
        for p in (1e-2, 2e-2):  # the second step of the same hierarchy
            pf.pressure_set(H, p)
            st = pf.rmtr_load_step(H, x, _params(pf, mixed, galerkin, rtol=1e-8))
            assert st["converged"] == 1
            runs.append((x.clone(), st["cycles"], st["cg"], st["energy"]))
        assert lib.probe_one_launch(H.handle) == 0
        out.append(runs)
        H.close()
    for a, b in zip(*out):
        assert torch.equal(a[0], b[0])
        assert a[1:] == b[1:]
