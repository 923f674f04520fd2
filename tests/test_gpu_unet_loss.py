"""The loss gradient dL/dy = (y - t) mask / n rounds the FP64 product once,
whatever the magnitudes: every bit of it against numpy, over the whole range of
FP32 (zeros, subnormal quotients and ones that leave the range included)."""
import numpy as np
import pytest

import pfinputs as PI
from tests.gpu_common import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("lo,hi", [(-20, 20), (-149, 127)])
def test_loss_gradient_is_rounded_once(masked, lo, hi):
    torch = require_cuda()
    from paper_2007_12908_gb300 import _binding as B
    h, w, c = 256, 392, 3
    r = PI.rng(17)
    y = np.ldexp(r.uniform(-1.0, 1.0, (c, h, w)), r.integers(lo, hi, (c, h, w))).astype(np.float32)
    y.reshape(-1)[::101] = 0.0
    y.reshape(-1)[5::103] = -0.0
    t = np.zeros_like(y)
    mask = (r.uniform(0.0, 1.0, (h, w)) < 0.7).astype(np.float32) if masked else np.ones((h, w), np.float32)
    n_valid = float(mask.sum())
    net = B.Unet(h, w, n_in=1, n_out=c, channels=(4, 4, 4, 4))
    args = [torch.from_numpy(a).cuda() for a in (y, t)]
    if masked:
        _, dy = net.mse(*args, mask=torch.from_numpy(mask).cuda(), n_valid=n_valid)
    else:
        _, dy = net.mse(*args)
    net.close()
    d = (y - t) * mask
    with np.errstate(over="ignore"):
        want = (d.astype(np.float64) * (1.0 / (c * n_valid))).astype(np.float32)
    assert np.array_equal(dy.cpu().numpy().view(np.uint32), want.view(np.uint32))
