"""Kernels that start while the launch before them drains give the bits of
launches that wait for one another: mixed 3D load steps (element-owned levels and
smaller ones, and GALERKIN coarse operators) in a process that blocks after every
launch, and a chain of transfers and Galerkin operators replayed from a captured
graph, whose launches are plain."""
import os
import subprocess
import sys

import pytest

import pfinputs as PI
from tests.gpu_common import dev, require_cuda

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STEP = """
import hashlib, sys
sys.path.insert(0, sys.argv[1])
import torch
import paper_2007_12908_gb300 as pf
import pfinputs as PI
for galerkin in (0, 1):
    H = pf.mesh_hierarchy_create(3, (15, 15, 15), 3, 1 / 14, E=1.0, nu=0.25, Gc=1.0)
    pf.pressure_set(H, 5e-3)
    x = torch.zeros(H.ndof(), dtype=torch.float64, device="cuda")
    pf.fractures_set(H, pf.PF_DISC3D, PI.disc_network_3d(PI.SEED_3D_PLAIN, 5), H.levels[-1][1], x)
    st = pf.rmtr_load_step(H, x, pf.default_params(precision=pf.PF_FP32, max_cycles=2, coarse_model=1 - galerkin),
                           check=False)
    print(galerkin, st["cg"], st["cycles"], hashlib.sha256(x.cpu().numpy().tobytes()).hexdigest())
"""


def _step(blocking):
    env = dict(os.environ, CUDA_LAUNCH_BLOCKING="1" if blocking else "0")
    r = subprocess.run([sys.executable, "-c", STEP, ROOT], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return r.stdout


def test_mixed_load_step():
    require_cuda()
    assert _step(False) == _step(True)


@pytest.mark.parametrize("nc", [(9, 7), (33, 30), (9, 7, 6), (33, 25, 29)])
def test_chain_of_transfers_and_galerkin(nc):
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        H = pf.mesh_hierarchy_create(len(nc), nc, 2, 1.0 / (max(nc) - 1), E=1.0, nu=0.25, Gc=1.0, stream=st)
        x32 = dev(PI.random_state(1, len(nc), H.nodes(), u_scale=1e-2), torch.float32)
        v = dev(PI.random_direction(2, H.ndof(0)))
        pf.galerkin_set(H, x32)  # allocates
        f = [torch.empty(H.ndof(1), dtype=torch.float64, device="cuda") for _ in range(2)]
        c = [torch.empty_like(v) for _ in range(4)]

        def chain(wait, capture=False):
            for k in range(2):
                for op, src, out in ((pf.galerkin_apply, v if k == 0 else c[3], c[0]), (pf.prolong, c[0], f[0]),
                                     (pf.restrict, f[0], c[1]), (pf.prolong, c[1], f[1]), (pf.project, f[1], c[2])):
                    op(H, 0, src, out)
                    if wait:
                        torch.cuda.synchronize()
                if not capture:  # it synchronises
                    pf.galerkin_set(H, x32)
                pf.galerkin_apply(H, 0, c[2], c[3])
            return torch.cat(c + f)

        want = chain(True).clone()
        got = [chain(False).clone() for _ in range(3)]
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        replayed = chain(False, capture=True)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.isfinite(want).all()
    assert all(torch.equal(want, g) for g in got)
    assert torch.equal(want, replayed)
    H.close()
