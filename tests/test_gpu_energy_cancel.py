"""The energy of one element where its quadratic terms cancel: displacements
that keep the volume near incompressibility (lam / mu up to 5e5) and that
nearly rotate the element, against 80-bit or wider arithmetic.  The error may
be that of rounded derivatives: eps times |lam tr| |G| + mu |strain| |G| + psi
summed over the Gauss points, with a factor 32 for the chain of operations
(double-float: eps 2^-46)."""
import numpy as np
import pytest

import pfinputs as PI
from tests.element_exact import energy_terms
from tests.gpu_common import dev, require_cuda

pytestmark = pytest.mark.gpu


def _displacement(kind, r, dim, h):
    a = r.standard_normal((dim, dim))
    if kind == "isochoric":
        a -= np.eye(dim) * np.trace(a) / dim
    else:
        a = a - a.T + 1e-4 * r.standard_normal((dim, dim))
    corners = np.array([[(k >> i) & 1 for i in range(dim)] for k in range(1 << dim)]) * h
    return 1e-3 * a @ corners.T


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind,nu", [("isochoric", 0.25), ("isochoric", 0.4999), ("isochoric", 0.499999),
                                     ("rotation", 0.25), ("rotation", -0.5)])
def test_energy_keeps_its_digits(dim, kind, nu):
    require_cuda()
    import paper_2007_12908_gb300 as pf
    h = 1.0 / 16.0
    H = pf.mesh_hierarchy_create(dim, (2,) * dim, 1, h, E=1.0, nu=nu, Gc=1e-12)
    pf.pressure_set(H, 0.0)
    r = PI.rng(41)
    for _ in range(20):
        x = np.concatenate([_displacement(kind, r, dim, h), r.uniform(0.0, 0.9, (1, 1 << dim))])
        exact, scale = energy_terms(dim, x, nu, 1e-12, h)
        d = dev(x.reshape(-1))
        assert abs(np.longdouble(pf.energy(H, 0, d)) - exact) <= 32 * 2.0**-53 * scale
        if dim == 3:  # the double-float scratch does not fit a single 2D element
            assert abs(np.longdouble(pf.energy_df(H, 0, d)) - exact) <= 32 * 2.0**-46 * scale
    H.close()
