"""The FP32 one-launch subproblem (stored Galerkin operators, rows held in
registers) against its FP64 form on the same numbers, at the edges of its split (a
warp, a CTA, the most rows), with and without the preconditioner and restarts, with
budgets that end in mid-run.  Decisions may fall differently at a tie, so the model
values are compared, within 1e-3 of each other; the step lies in the box."""
import ctypes as C

import numpy as np
import pytest

import pfinputs as PI
from tests.gpu_common import dev, host, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,cg,restarts,pre", [
    ((3, 3), 12, 100, True), ((40, 40), 12, 100, True), ((41, 40), 5, 100, False), ((113, 114), 12, 0, True),
    ((5, 4, 3), 12, 100, True), ((23, 21, 20), 8, 100, True), ((32, 19, 16), 8, 0, False), ((9, 8, 7), 60, 100, False),
])
def test_against_fp64(nc, cg, restarts, pre):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    from tests import native_probe as probe
    lib = probe.load()
    dim = len(nc)
    H = pf.mesh_hierarchy_create(dim, nc, 2, 1.0 / (max(nc) - 1), E=1.0, nu=0.25, Gc=1.0)
    pf.pressure_set(H, 1e-2)
    pf.galerkin_set(H, dev(PI.random_state(3, dim, H.nodes(), u_scale=1e-2), torch.float32))
    n, F = H.ndof(0), dim + 1
    S32 = torch.empty(3**dim * F * n, dtype=torch.float32, device="cuda")
    assert lib.probe_galerkin_stencil(H.handle, C.c_int(0), probe.ptr(S32)) == 0
    N = H.nodes(0)
    centre = S32.view(3**dim, F, F, N)[3**dim // 2]
    diag = torch.stack([centre[f, f] for f in range(F)]).reshape(-1)
    assert bool((diag > 0).all())
    # a gradient whose Newton step leaves the box in about half of its dofs
    g = diag.double() * dev(PI.random_direction(4, n))
    lo, hi = dev(-PI.rng(5).uniform(0.0, 1.0, n)), dev(PI.rng(6).uniform(0.0, 1.0, n))
    m, out = [], []
    for fp32, dt in ((1, torch.float32), (0, torch.float64)):
        S, mi = S32.to(dt), (1.0 / diag).to(dt)
        s = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
        stats = (C.c_int * 2)()
        rc = lib.probe_subproblem(H.handle, C.c_int(0), C.c_int(fp32), probe.ptr(S), probe.ptr(mi if pre else None),
                                  probe.ptr(g), probe.ptr(lo), probe.ptr(hi), probe.ptr(s), C.c_int(cg),
                                  C.c_int(restarts), stats)
        assert rc == 0
        sh = host(s)
        assert np.all(sh >= host(lo)) and np.all(sh <= host(hi))
        assert 0 < stats[0] <= cg and stats[1] <= restarts + 1
        m.append(float(torch.dot(g, s) + 0.5 * torch.dot(s, pf.galerkin_apply(H, 0, s))))
        out.append(list(stats))
    H.close()
    assert m[1] < 0.0
    assert abs(m[0] - m[1]) <= 1e-3 * abs(m[1]), (m, out)
