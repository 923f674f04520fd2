"""One Q1 element of the pressurised AT2 functional in numpy's widest float, by
sums over the Gauss points (k = 0, l_s = 2 h), for the tests of rounding
errors.  States are (dim + 1, 2^dim) corner values."""
import numpy as np

W = np.longdouble


def _shapes(dim):
    xi = [(1 - 1 / np.sqrt(W(3))) / 2, (1 + 1 / np.sqrt(W(3))) / 2]
    nc = 1 << dim
    n = np.ones((nc, nc), W)
    g = np.ones((dim, nc, nc), W)
    for q in range(nc):
        for a in range(nc):
            for k in range(dim):
                t, b = xi[(q >> k) & 1], (a >> k) & 1
                v = t if b else 1 - t
                n[q, a] *= v
                for j in range(dim):
                    g[j, q, a] *= (W(1) if b else W(-1)) if j == k else v
    return n, g


def _lame(nu, E):
    return W(E) * W(nu) / ((1 + W(nu)) * (1 - 2 * W(nu))), W(E) / (2 * (1 + W(nu)))


def _fields(dim, x, h):
    n, g = _shapes(dim)
    x = x.astype(W)
    grad = np.einsum("kqa,...ia->...ikq", g, x[..., :dim, :]) / W(h)
    return n, g, grad, x[..., dim, :] @ n.T, np.einsum("kqa,...a->...kq", g, x[..., dim, :]) / W(h)


def _psi(dim, grad, lam, mu, p):
    tr = sum(grad[..., i, i, :] for i in range(dim))
    e = (grad + np.swapaxes(grad, -3, -2)) / 2
    return tr, e, lam / 2 * tr * tr + mu * (e * e).sum((-3, -2)) + p * tr


def energy_terms(dim, x, nu, Gc, h, p=0.0, E=1.0):
    """The energy, and the magnitude of what its rounding is relative to."""
    lam, mu = _lame(nu, E)
    _, _, grad, c, gc = _fields(dim, x, h)
    tr, e, psi = _psi(dim, grad, lam, mu, W(p))
    w, ls = W(h) ** dim / 2**dim, 2 * W(h)
    g = (1 - c) ** 2
    frac = W(Gc) / 2 * (c * c / ls + ls * (gc * gc).sum(-2))
    size = np.sqrt((grad * grad).sum((-3, -2)))
    strain = np.sqrt((e * e).sum((-3, -2)))
    scale = g * (abs(lam * tr) * size + 2 * mu * strain * size + abs(psi)) + frac
    return (w * (g * psi + frac)).sum(-1), (w * scale).sum(-1)


def gradient(dim, x, nu, Gc, h, p=0.0, E=1.0):
    """The gradient by corner, like x."""
    lam, mu = _lame(nu, E)
    n, s, grad, c, gc = _fields(dim, x, h)
    tr, e, psi = _psi(dim, grad, lam, mu, W(p))
    w, ls = W(h) ** dim / 2**dim, 2 * W(h)
    stress = 2 * mu * e + np.eye(dim, dtype=W)[:, :, None] * (lam * tr + W(p))[..., None, None, :]
    out = np.empty(x.shape, W)
    out[..., :dim, :] = np.einsum("...ikq,...q,kqa->...ia", stress, (1 - c) ** 2 * w / W(h), s)
    out[..., dim, :] = (w * (W(Gc) / ls * c - 2 * (1 - c) * psi)) @ n
    out[..., dim, :] += np.einsum("...kq,kqa->...a", gc * (w * W(Gc) * ls / W(h)), s)
    return out


def hessvec(dim, x, v, nu, Gc, h, p=0.0, E=1.0):
    """The Hessian at x applied to v."""
    lam, mu = _lame(nu, E)
    n, s, grad, c, _ = _fields(dim, x, h)
    _, _, gv, wv, gw = _fields(dim, v, h)
    tr, e, psi = _psi(dim, grad, lam, mu, W(p))
    trv, ev, _ = _psi(dim, gv, lam, mu, W(0))
    w, ls = W(h) ** dim / 2**dim, 2 * W(h)
    eye = np.eye(dim, dtype=W)[:, :, None]
    stress = 2 * mu * e + eye * (lam * tr + W(p))[..., None, None, :]
    g, dg = (1 - c) ** 2, -2 * (1 - c)
    su = (2 * mu * ev + eye * (lam * trv)[..., None, None, :]) * g[..., None, None, :]
    su = su + stress * (dg * wv)[..., None, None, :]
    out = np.empty(x.shape, W)
    out[..., :dim, :] = np.einsum("...ikq,kqa->...ia", su * (w / W(h)), s)
    out[..., dim, :] = (w * (dg * (stress * ev).sum((-3, -2)) + (2 * psi + W(Gc) / ls) * wv)) @ n
    out[..., dim, :] += np.einsum("...kq,kqa->...a", gw * (w * W(Gc) * ls / W(h)), s)
    return out
