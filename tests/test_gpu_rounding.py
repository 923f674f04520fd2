"""Rounding errors of the element passes on single 3D elements with rough
displacements (independent corner values, lam = mu = 1, a toughness of 2^-40 so
that the displacement terms decide), as root mean square over many elements
against 80-bit or wider arithmetic.  LIMIT is what the evaluation axis by axis
has there, every Gauss value formed as v + xi d with fused multiply-adds (4,000
elements), and 7 % for the sampling."""
import numpy as np
import pytest

import pfinputs as PI
from tests import element_exact as X
from tests.gpu_common import require_cuda

pytestmark = pytest.mark.gpu

E, NU, GC, H1, N = 2.5, 0.25, 2.0**-40, 1.0 / 16.0, 2000
LIMIT = {"energy": 1.52e-16, "gradient u": 2.08e-16, "gradient c": 1.93e-16,
         "energy df": 3.87e-15, "gradient df u": 5.45e-15, "gradient df c": 4.37e-15,
         "product u": 1.06e-7, "product c": 1.57e-7}


def _states(seed, n):
    r = PI.rng(seed)
    return np.concatenate([1e-3 * r.standard_normal((n, 3, 8)), r.uniform(0.0, 1.0, (n, 1, 8))], axis=1)


def _rms(got, exact, rows):
    d = (got[:, rows].astype(X.W) - exact[:, rows]).reshape(len(got), -1)
    e = exact[:, rows].reshape(len(got), -1)
    return float(np.sqrt(np.mean((d * d).sum(1) / (e * e).sum(1))))


def _element(pf):
    H = pf.mesh_hierarchy_create(3, (2, 2, 2), 1, H1, E=E, nu=NU, Gc=GC)
    pf.pressure_set(H, 0.0)
    return H


def test_energy_and_gradient():
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H = _element(pf)
    x = _states(51, N)
    xd = torch.from_numpy(x.reshape(N, -1)).cuda()
    energy, _ = X.energy_terms(3, x, NU, GC, H1, E=E)
    grad = X.gradient(3, x, NU, GC, H1, E=E)
    got = {}
    for name, ef, gf in (("", pf.energy, pf.gradient), (" df", pf.energy_df, pf.gradient_df)):
        e = np.array([ef(H, 0, v) for v in xd])
        g = torch.stack([gf(H, 0, v) for v in xd]).cpu().numpy().reshape(x.shape)
        got["energy" + name] = _rms(e[:, None], energy[:, None], slice(None))
        got["gradient" + name + " u"] = _rms(g, grad, slice(0, 3))
        got["gradient" + name + " c"] = _rms(g, grad, slice(3, 4))
    H.close()
    assert all(got[k] <= 1.07 * LIMIT[k] for k in got), got


def test_fp32_product():
    torch = require_cuda()
    import paper_2007_12908_gb300 as pf
    H = _element(pf)
    x = _states(53, N).astype(np.float32)
    v = PI.rng(54).standard_normal(x.shape).astype(np.float32)
    xd, vd = torch.from_numpy(x.reshape(N, -1)).cuda(), torch.from_numpy(v.reshape(N, -1)).cuda()
    exact = X.hessvec(3, x, v, NU, GC, H1, E=E)
    y = torch.stack([pf.hessvec(H, 0, a, b) for a, b in zip(xd, vd)]).cpu().numpy().reshape(x.shape)
    H.close()
    got = {"product u": _rms(y, exact, slice(0, 3)), "product c": _rms(y, exact, slice(3, 4))}
    assert all(got[k] <= 1.07 * LIMIT[k] for k in got), got
