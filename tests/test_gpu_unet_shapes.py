"""The U-Net's convolution kernels at the edges of their tiles (16 x 8 pixels,
16 x 16 in the weight gradient), of their channel padding (16) and over all
channel blocks, against the same network in torch FP64 with every stored value
rounded to BF16 as the library stores it (inputs, weights, activations and
pooled activations).  The biases keep every ReLU open: with masks that flip
where a pre-activation is within rounding of 0, the gradients of two correct
implementations differ by several per cent on these small grids (masks are
compared with the oracle in test_gpu_unet.py on 64 x 64).  What is left between
the two sides is FP32 accumulation, which moves a stored value to the next BF16
number now and then, 2^-8 of it: relative L2 within 2^-8."""
import numpy as np
import pytest

from tests.gpu_common import require_cuda

pytestmark = pytest.mark.gpu


def _shapes(n_in, n_out, ch):
    out, c = [], n_in
    for k in range(4):
        out += [(ch[k], c, 3), (ch[k], ch[k], 3)]
        c = ch[k]
    for k in (2, 1, 0):
        out += [(ch[k], ch[k + 1] + ch[k], 3), (ch[k], ch[k], 3)]
    return out + [(n_out, ch[0], 1)]


def _reference(torch, flat, shapes, x):
    F = torch.nn.functional

    def stored(t):  # BF16 value, gradient passed through
        return t + (t.detach().to(torch.bfloat16).double() - t.detach())

    ws, off = [], 0
    for co, ci, k in shapes:
        n = co * ci * k * k
        ws.append((stored(flat[off:off + n].reshape(co, ci, k, k)), flat[off + n:off + n + co]))
        off += n + co

    def conv(t, i):
        w, b = ws[i]
        return F.conv2d(t, w, b, padding=w.shape[-1] // 2)

    t, skips = stored(x)[None], []
    for k in range(4):
        if k:
            t = stored(F.avg_pool2d(t, 2))
        t = stored(torch.relu(conv(t, 2 * k)))
        t = stored(torch.relu(conv(t, 2 * k + 1)))
        skips.append(t)
    for d, k in enumerate((2, 1, 0)):
        t = torch.cat([t.repeat_interleave(2, 2).repeat_interleave(2, 3), skips[k]], 1)
        t = stored(torch.relu(conv(t, 8 + 2 * d)))
        t = stored(torch.relu(conv(t, 9 + 2 * d)))
    return conv(t, 14)[0]


@pytest.mark.parametrize("H,W,n_in,n_out,ch", [
    (8, 8, 1, 1, (1, 2, 3, 4)), (16, 24, 5, 3, (16, 32, 64, 128)), (40, 8, 3, 2, (5, 9, 17, 33)),
    (24, 136, 17, 20, (16, 16, 48, 64)), (136, 40, 5, 3, (8, 40, 24, 16)), (512, 520, 5, 3, (16, 32, 64, 128))])
def test_unet_matches_stored_precision_reference(H, W, n_in, n_out, ch):
    torch = require_cuda()
    from paper_2007_12908_gb300 import _binding as B
    shapes = _shapes(n_in, n_out, ch)
    r = np.random.default_rng(H * 1000 + W)
    flat = np.concatenate([np.concatenate([r.standard_normal(co * ci * k * k) * 0.1 / np.sqrt(ci * k * k),
                                           0.1 * r.standard_normal(co) + 2.0])
                           for co, ci, k in shapes]).astype(np.float32)
    x = torch.from_numpy(r.standard_normal((n_in, H, W)).astype(np.float32)).cuda()
    dy = torch.from_numpy(r.standard_normal((n_out, H, W)).astype(np.float32)).cuda()
    net = B.Unet(H, W, n_in, n_out, ch)
    assert net.n_params == flat.size
    net.set_params(flat)
    y = net.forward(x)
    net.backward(dy)
    g1 = net.get_grads()
    net.set_params(flat)
    assert torch.equal(net.forward(x), y)
    net.backward(dy)
    assert np.array_equal(net.get_grads(), g1)  # deterministic
    f = torch.from_numpy(flat).cuda().double().requires_grad_(True)
    yo = _reference(torch, f, shapes, x.double())
    go, = torch.autograd.grad((yo * dy.double()).sum(), f)
    go = go.cpu().numpy()

    def rel(a, b):
        return float(np.linalg.norm(a - b) / np.linalg.norm(b))

    assert rel(y.double().cpu().numpy().ravel(), yo.detach().cpu().numpy().ravel()) <= 2.0 ** -8
    assert rel(g1.astype(np.float64), go) <= 2.0 ** -8
    # a second backward adds to the gradient
    net.backward(dy)
    assert rel(net.get_grads().astype(np.float64), 2 * g1.astype(np.float64)) <= 1e-6
    net.close()
