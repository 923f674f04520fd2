"""The work a user of this framework has it do, as cases that can be timed and
compared: load steps, the operators a solver is written with, the batched
operators and the learned initial iterate, each through the package's public
calls, from the smallest grids (launches and latency) to the largest.

Sizes are those of the tests and the benchmark (65^2 and 1025^2 in 2D, 17^3 to
129^3 in 3D, the 129^2 to 1025^2 batch, the 129^2 learned workload) and ragged
ones in between.  `nodes` counts nodes per axis, x first.

Kinds:
  step       one load step of a fractured medium from its initial state: the
             call the library exists for (FP64 with the default parameters, or
             mixed precision)
  newton     what a second-order method of the user's own asks for at one
             iterate, in FP64: energy, gradient, a lagged Hessian and its
             product with several directions
  product    one FP32 Hessian-vector product, the inner step of any Krylov
             method on the functional
  stopping   gradient and energy of an FP64 state in double-float arithmetic:
             the stopping test of a mixed-precision solver
  transfer   one coarse start of a multilevel method: the projected iterate,
             the restricted gradient, the coarse bounds and the prolonged
             correction
  galerkin   the stored Galerkin operators of every coarse level from a new
             lag point, and one product on each
  batch      Hessian products and energies of many networks of uneven size
  propose    the learned iterate's inference: features, network, proposal
  train      loss and parameter gradient of the network over a few samples
"""
import math

import numpy as np
import torch
import torch.nn.functional as nnf

import paper_2007_12908_gb300 as pf
from paper_2007_12908_gb300 import _binding as pfb
from paper_2007_12908_gb300 import learned

XI = ((1.0 - 1.0 / math.sqrt(3.0)) / 2.0, (1.0 + 1.0 / math.sqrt(3.0)) / 2.0)
NU = 0.25
DIRECTIONS = 8  # lagged products per lag in the newton kind
E_MOD, GC, LS_OVER_H = 1.0, 1.0, 2.0


def listed():
    return [
        # the smallest whole solve: the 2D centred-crack workload's grid, FP64
        # with the default parameters (tests, smoke runs, first experiments)
        {"name": "step_2d_65_fp64", "kind": "step", "nodes": "65x65", "levels": 2, "fp32": False, "cracks": 1},
        # the 3D workload: first ramp step of 20 discs at 129^3, mixed precision
        {"name": "step_3d_129_mixed", "kind": "step", "nodes": "129x129x129", "levels": 4, "fp32": True, "cracks": 20},
        # a user's own Newton or trust-region loop on a small 2D grid, ragged
        {"name": "newton_2d_69x45", "kind": "newton", "nodes": "69x45"},
        # the same in 3D, where the FP64 Hessian is assembled and streamed
        {"name": "newton_3d_65x49x57", "kind": "newton", "nodes": "65x49x57"},
        # the product that carries the mixed-precision solver, at full size
        {"name": "product_3d_129", "kind": "product", "nodes": "129x129x129"},
        # and on a coarse level, where one launch is all there is
        {"name": "product_3d_33x25x29", "kind": "product", "nodes": "33x25x29"},
        # the mixed solver's stopping test on an odd grid
        {"name": "stopping_3d_97x105x89", "kind": "stopping", "nodes": "97x105x89"},
        # the transfers between the two finest levels of the 3D workload
        {"name": "transfer_3d_129", "kind": "transfer", "nodes": "129x129x129"},
        # the second-order coarse models of a three-level 3D hierarchy
        {"name": "galerkin_3d_65", "kind": "galerkin", "nodes": "65x65x65", "levels": 3},
        # an uneven batch of fracture networks (one quarter of the 64-instance draw)
        {"name": "batch_2d_16", "kind": "batch", "instances": 16, "largest": 1025},
        # the learned workload's test size: one proposal per load step
        {"name": "propose_129", "kind": "propose", "nodes": "129x129"},
        # training on a 4x larger, ragged grid (padded to 528 x 520)
        {"name": "train_513x521", "kind": "train", "nodes": "513x521", "samples": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "newton", "product", "stopping", "transfer", "galerkin", "batch",
                       "propose", "train"])
    dim = rng.choice([2, 3])

    def nodes(lo2, hi2, lo3, hi3, step=1, odd=0):
        out = []
        base = _log(rng, lo2, hi2) if dim == 2 else _log(rng, lo3, hi3)
        for _ in range(dim):
            n = max(4, int(base * rng.uniform(0.7, 1.0)))
            out.append((n - odd) // step * step + odd if step > 1 else n)
        return "x".join(str(max(n, step + odd, 4)) for n in out)

    if kind == "step":
        fp32 = rng.choice([False, True])
        if dim == 2:
            levels = rng.choice([2, 3])
            n = nodes(40, 240, 0, 0, 1 << (levels - 1), 1)
            return {"kind": "step", "nodes": n, "levels": levels, "fp32": fp32, "cracks": rng.randint(1, 4)}
        levels = rng.choice([2, 3])
        n = nodes(0, 0, 20, 120 if fp32 else 56, 1 << (levels - 1), 1)
        return {"kind": "step", "nodes": n, "levels": levels, "fp32": fp32, "cracks": rng.randint(2, 20)}
    if kind == "newton":
        return {"kind": "newton", "nodes": nodes(17, 513, 9, 65)}
    if kind == "product":
        return {"kind": "product", "nodes": nodes(65, 1025, 17, 129)}
    if kind == "stopping":
        return {"kind": "stopping", "nodes": nodes(65, 1025, 17, 129)}
    if kind == "transfer":
        return {"kind": "transfer", "nodes": nodes(65, 1025, 17, 129, 2, 1)}
    if kind == "galerkin":
        levels = rng.choice([2, 3])
        return {"kind": "galerkin", "nodes": nodes(65, 513, 17, 65, 1 << (levels - 1), 1), "levels": levels}
    if kind == "batch":
        return {"kind": "batch", "instances": rng.randint(3, 16), "largest": _log(rng, 129, 1025)}
    dim = 2
    if kind == "propose":
        return {"kind": "propose", "nodes": nodes(65, 1025, 0, 0)}
    return {"kind": "train", "nodes": nodes(65, 700, 0, 0), "samples": rng.randint(1, 2)}


# ------------------------------------------------------------------ inputs
def _shape(case):
    return tuple(int(v) for v in case["nodes"].split("x"))


def _batch_shapes(case):
    """Nodes per axis of every instance: the sizes halve from the largest,
    an equal number of each, with ragged heights."""
    out = []
    for k in range(case["instances"]):
        nx = max(17, (case["largest"] - 1) // (1 << (k % 4)) + 1)
        out.append((nx, max(9, nx - 13 * (k // 4))))
    return out


def _count(n):
    return int(np.prod(n))


def _elements(n):
    return int(np.prod([v - 1 for v in n]))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _cracked_state(n, h, seed, cracks=6):
    """A state as a load step meets it: displacements of the size the pressure
    of 5e-4 opens cracks by, a phase field decaying from a few cracks (1 on
    their mid-surfaces), and a little of everything everywhere."""
    dim, g = len(n), _gen(seed)
    axes = [torch.arange(m, dtype=torch.float64, device="cuda") * h for m in n]
    grid = torch.meshgrid(*reversed(axes), indexing="ij")
    X = [a.reshape(-1) for a in reversed(grid)]
    size = [float((m - 1) * h) for m in n]
    c = torch.zeros_like(X[0])
    for _ in range(cracks):
        r = torch.rand(2 * dim + 1, dtype=torch.float64, device="cuda", generator=g)
        normal = torch.randn(dim, dtype=torch.float64, device="cuda", generator=g)
        normal = normal / normal.norm()
        d = [X[k] - r[k] * size[k] for k in range(dim)]
        dn = sum(d[k] * normal[k] for k in range(dim))
        rad = sum((d[k] - dn * normal[k]) ** 2 for k in range(dim)).sqrt()
        over = (rad - (0.05 + 0.1 * r[-1])).clamp_min(0.0)
        dist = ((dn.abs() - h).clamp_min(0.0) ** 2 + over ** 2).sqrt()
        c = torch.maximum(c, torch.exp(-dist / (LS_OVER_H * h)))
    x = torch.empty((dim + 1, c.numel()), dtype=torch.float64, device="cuda")
    for k in range(dim):
        ph = torch.rand(dim + 1, dtype=torch.float64, device="cuda", generator=g) * 6.0
        wave = torch.ones_like(c)
        for j in range(dim):
            wave = wave * torch.sin(4.0 * X[j] + ph[j])
        noise = torch.rand(c.shape, dtype=torch.float64, device="cuda", generator=g) - 0.5
        x[k] = 1e-4 * wave + 1e-6 * noise
    noise = torch.rand(c.shape, dtype=torch.float64, device="cuda", generator=g)
    x[dim] = torch.clamp(c * (1.0 - 1e-3 * noise), 0.0, 1.0)
    return x.reshape(-1)


def _direction(n, seed):
    """A search direction: displacement and phase-field parts of their own
    sizes, zero displacement on the clamped boundary."""
    dim = len(n)
    v = torch.randn((dim + 1,) + tuple(reversed(n)), dtype=torch.float64, device="cuda", generator=_gen(seed))
    v[:dim] *= 1e-2
    for k in range(dim):
        ax = dim - k  # x is the last axis
        for i in (0, n[k] - 1):
            v[:dim].select(ax, i).zero_()
    return v.reshape(-1)


def _hierarchy(n, levels=1):
    f = 1 << (levels - 1)
    coarse = [(m - 1) // f + 1 for m in n]
    h = 1.0 / (max(n) - 1)
    H = pf.mesh_hierarchy_create(len(n), coarse, levels, h * f, E=E_MOD, nu=NU, Gc=GC, ls_over_h=LS_OVER_H)
    return H, h


def _crack_rows(dim, cracks, seed):
    rng = np.random.default_rng(int(seed))
    rows = []
    for _ in range(cracks):
        cen = rng.uniform(0.25, 0.75, size=dim)
        if dim == 2:
            rows.append([cen[0], cen[1], rng.uniform(-0.6, 0.6), rng.uniform(0.05, 0.12)])
        else:
            nv = rng.standard_normal(3)
            rows.append(list(rng.uniform(0.0, 1.0, size=3)) + list(nv / np.linalg.norm(nv)) + [rng.uniform(0.03, 0.1)])
    return np.array(rows)


def _params(seed, shapes):
    """He-normal weights with small random biases and a small random head."""
    rng = np.random.default_rng(int(seed))
    parts = []
    for i, (co, ci, k) in enumerate(shapes):
        scale = 1.0 if i < len(shapes) - 1 else 0.3
        parts.append(rng.standard_normal(co * ci * k * k) * (scale * math.sqrt(2.0 / (ci * k * k))))
        parts.append(0.05 * rng.standard_normal(co))
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    p = 5e-4
    if kind == "batch":
        s["Hs"], s["x"], s["v"], s["y"], s["x64"] = [], [], [], [], []
        for k, n in enumerate(_batch_shapes(case)):
            H, h = _hierarchy(n)
            pf.pressure_set(H, p * (1 + k % 3))
            x = _cracked_state(n, h, seed * 1000 + 2 * k)
            s["Hs"].append(H)
            s["x64"].append(x)
            s["x"].append(x.float())
            s["v"].append(_direction(n, seed * 1000 + 2 * k + 1).float())
            s["y"].append(torch.empty_like(s["v"][-1]))
        s["batch"] = pf.Batch(s["Hs"])
        return s
    n = _shape(case)
    H, h = _hierarchy(n, case.get("levels", 2 if kind == "transfer" else 1))
    top = H.n_levels - 1
    s.update(H=H, top=top)
    if kind == "step":
        x0 = torch.zeros(H.ndof(), dtype=torch.float64, device="cuda")
        pf.fractures_set(H, pf.PF_LINE2D if len(n) == 2 else pf.PF_DISC3D,
                         _crack_rows(len(n), case["cracks"], seed), h, x0)
        s.update(x0=x0, x=torch.empty_like(x0), p=p,
                 params=pf.default_params(rtol=1e-12, precision=pf.PF_FP32 if case["fp32"] else pf.PF_FP64))
        return s
    pf.pressure_set(H, p)
    x = _cracked_state(n, h, seed)
    if kind == "newton":
        v = [_direction(n, seed * 100 + k) for k in range(DIRECTIONS)]
        s.update(x=x, g=torch.empty_like(x), v=v, hv=[torch.empty_like(x) for _ in v])
    elif kind == "product":
        s.update(x=x.float(), v=_direction(n, seed + 1).float())
        s["hv"] = torch.empty_like(s["v"])
    elif kind == "stopping":
        s.update(x=x, g=torch.empty_like(x))
    elif kind == "transfer":
        N, dim = H.nodes(), len(n)
        lo = torch.full_like(x, -1.0)
        hi = torch.ones_like(x)
        lo[dim * N:] = 0.0
        hi[dim * N:] = 1.0 - x[dim * N:]
        nc = H.ndof(0)
        s.update(x=x, g=_direction(n, seed + 1), lo=lo, hi=hi,
                 sc=torch.randn(nc, dtype=torch.float64, device="cuda", generator=_gen(seed + 2)),
                 xc=torch.empty(nc, dtype=torch.float64, device="cuda"),
                 gc=torch.empty(nc, dtype=torch.float64, device="cuda"), sf=torch.empty_like(x))
    elif kind == "galerkin":
        v = [torch.randn(H.ndof(l), device="cuda", generator=_gen(seed + 1 + l)) for l in range(top)]
        s.update(x=x.float(), v=v, hv=[torch.empty_like(t) for t in v])
    elif kind == "propose":
        L = learned.LearnedIterate(H)
        L.net.set_params(_params(seed + 7, learned.layer_shapes()))
        N = H.nodes()
        c_before = (x[2 * N:] * 0.98).clone()
        s.update(L=L, x=x, c_before=c_before, p_prev=p, p_new=1.5 * p,
                 y=torch.empty((3, L.Hp, L.Wp), device="cuda"), xhat=torch.empty_like(x))
    elif kind == "train":
        L = learned.LearnedIterate(H)
        s.update(L=L, flat=_params(seed + 7, learned.layer_shapes()), data=[])
        g = _gen(seed + 3)
        for _ in range(case["samples"]):
            f = torch.randn((5, L.Hp, L.Wp), device="cuda", generator=g)
            t = torch.randn((3, L.Hp, L.Wp), device="cuda", generator=g)
            s["data"].append((f * L.mask, t * L.mask))
    return s


# ------------------------------------------------------------------ the calls
def run(s):
    kind = s["kind"]
    if kind == "step":
        s["x"].copy_(s["x0"])
        pf.pressure_set(s["H"], s["p"])
        st = pf.rmtr_load_step(s["H"], s["x"], s["params"])
        return {"x": s["x"], "energy": st["energy"]}
    if kind == "newton":
        H, top = s["H"], s["top"]
        e = pf.energy(H, top, s["x"])
        pf.gradient(H, top, s["x"], s["g"])
        pf.hessvec_lag_set(H, top, s["x"])
        for v, o in zip(s["v"], s["hv"]):
            pf.hessvec_lagged(H, top, v, o)
        return {"energy": e, "gradient": s["g"], "hv": s["hv"]}
    if kind == "product":
        return pf.hessvec(s["H"], s["top"], s["x"], s["v"], s["hv"])
    if kind == "stopping":
        pf.gradient_df(s["H"], s["top"], s["x"], s["g"])
        return {"gradient": s["g"], "energy": pf.energy_df(s["H"], s["top"], s["x"])}
    if kind == "transfer":
        H = s["H"]
        pf.project(H, 0, s["x"], s["xc"])
        pf.restrict(H, 0, s["g"], s["gc"])
        lo, hi = pf.coarse_bounds(H, 0, s["lo"], s["hi"])
        pf.prolong(H, 0, s["sc"], s["sf"])
        return {"x": s["xc"], "g": s["gc"], "lo": lo, "hi": hi, "s": s["sf"]}
    if kind == "galerkin":
        pf.galerkin_set(s["H"], s["x"])
        for l, (v, o) in enumerate(zip(s["v"], s["hv"])):
            pf.galerkin_apply(s["H"], l, v, o)
        return s["hv"]
    if kind == "batch":
        s["batch"].hessvec(s["x"], s["v"], s["y"])
        return {"hv": s["y"], "energy": s["batch"].energy(s["x64"])}
    L = s["L"]
    if kind == "propose":
        f = L.features(s["x"], s["c_before"], s["p_prev"], s["p_new"])
        L.net.forward(f, s["y"])
        pfb.learned_apply(s["H"], s["x"], s["y"], s["p_prev"], s["p_new"], s["xhat"])
        return {"y": s["y"], "xhat": s["xhat"]}
    L.net.set_params(s["flat"])
    ys, losses = [], []
    for f, t in s["data"]:
        y = L.net.forward(f)
        loss, dy = L.net.mse(y, t, L.mask, L.n_valid)
        L.net.backward(dy)
        ys.append(y)
        losses.append(loss)
    return {"y": ys, "loss": losses, "grads": L.net.get_grads()}


# ------------------------------------------------------------------ necessary work
def work(case):
    """Inputs read once, outputs written once; operations of the element
    algebra (about 2,060 / 620 per element and Hessian product in 3D / 2D,
    the gradient and the energy roughly a half and a third of that), of the
    stencils and of the network's convolutions."""
    kind = case["kind"]
    if kind == "batch":
        n = [_count(v) for v in _batch_shapes(case)]
        el = [_elements(v) for v in _batch_shapes(case)]
        return {"bytes": sum(n) * 3 * (12 + 8), "flops": sum(el) * (620 + 200)}
    n = _shape(case)
    dim, N, NE = len(n), _count(n), _elements(n)
    nd = (dim + 1) * N
    hv, gr, en = ((2060, 1000, 700) if dim == 3 else (620, 310, 200))
    pts = 27 if dim == 3 else 9
    if kind == "step":
        # state in and out; two V-cycles of two smoothing steps of 50 CG
        # iterations are the least such a step has taken
        return {"bytes": 16 * nd, "flops": 200 * hv * NE}
    if kind == "newton":
        return {"bytes": 8 * nd * (2 + 2 * DIRECTIONS),
                "flops": (gr + en) * NE + DIRECTIONS * 2 * pts * (dim + 1) ** 2 * N}
    if kind == "product":
        return {"bytes": 12 * nd, "flops": hv * NE}
    if kind == "stopping":
        return {"bytes": 16 * nd, "flops": (gr + en) * NE}
    if kind == "transfer":
        nc = (dim + 1) * _count([(v - 1) // 2 + 1 for v in n])
        return {"bytes": 8 * (5 * nd + 5 * nc), "flops": 4 * 2 * nd}
    if kind == "galerkin":
        out, flops = 4 * nd, hv * NE
        for l in range(1, case["levels"]):
            c = _count([(v - 1) // (1 << l) + 1 for v in n])
            out += 8 * (dim + 1) * c
            flops += 2 * pts * (dim + 1) ** 2 * c
        return {"bytes": out, "flops": flops}
    Hp, Wp = learned.padded(n[1]), learned.padded(n[0])
    flops, b = 0, 0
    for i, (co, ci, k) in enumerate(learned.layer_shapes()):
        lev = i // 2 if i < 8 else (2 - (i - 8) // 2 if i < 14 else 0)
        flops += 2 * co * ci * k * k * (Hp * Wp >> (2 * lev))
        b += co * ci * k * k + co
    if kind == "propose":
        return {"bytes": 2 * b + 4 * 3 * Hp * Wp + 8 * (2 * nd + N), "flops": flops}
    return {"bytes": 8 * b + case["samples"] * 4 * (5 + 3 + 3) * Hp * Wp, "flops": 3 * flops * case["samples"]}


# ------------------------------------------------------------------ 64-bit values
class _Functional:
    """The discrete pressurised AT2 functional on one grid, in plain torch."""

    def __init__(self, n, h, ls, p):
        self.n, self.h, self.dim, self.p, self.ls = n, h, len(n), p, ls
        self.lam = E_MOD * NU / ((1 + NU) * (1 - 2 * NU))
        self.mu = E_MOD / (2 * (1 + NU))

    def _at(self, fields, q):
        """Values and gradients of all fields at Gauss point q of every element."""
        dim = self.dim
        val, grad = 0, [0] * dim
        for a in range(1 << dim):
            sl = [slice(None)]
            w, dw = 1.0, [1.0] * dim
            for k in reversed(range(dim)):  # tensors are (field, [z,] y, x)
                ak = (a >> k) & 1
                sl.append(slice(1, None) if ak else slice(0, -1))
                xi = XI[(q >> k) & 1]
                N = xi if ak else 1 - xi
                w *= N
                for j in range(dim):
                    dw[j] *= (1 if ak else -1) / self.h if j == k else N
            part = fields[tuple(sl)]
            val = val + w * part
            for j in range(dim):
                grad[j] = grad[j] + dw[j] * part
        return val, grad

    def energy_at(self, x, q):
        dim = self.dim
        val, grad = self._at(x.reshape((dim + 1,) + tuple(reversed(self.n))), q)
        c = val[dim]
        tr = sum(grad[i][i] for i in range(dim))
        ee = sum((0.5 * (grad[k][i] + grad[i][k])) ** 2 for i in range(dim) for k in range(dim))
        g = (1 - c) ** 2
        gc2 = sum(grad[k][dim] ** 2 for k in range(dim))
        dens = g * (0.5 * self.lam * tr * tr + self.mu * ee + self.p * tr)
        dens = dens + 0.5 * GC * (c * c / self.ls + self.ls * gc2)
        return dens.sum() * (self.h / 2) ** dim

    def energy(self, x):
        return float(sum(self.energy_at(x, q) for q in range(1 << self.dim)))

    def gradient(self, x):
        x = x.detach().requires_grad_(True)
        out = torch.zeros_like(x)
        for q in range(1 << self.dim):
            out += torch.autograd.grad(self.energy_at(x, q), x)[0]
        return out

    def hessvec(self, x, v):
        x = x.detach().requires_grad_(True)
        out = torch.zeros_like(x)
        for q in range(1 << self.dim):
            g, = torch.autograd.grad(self.energy_at(x, q), x, create_graph=True)
            out += torch.autograd.grad(g, x, grad_outputs=v)[0]
        return out


def _along(t, ax, sl):
    idx = [slice(None)] * t.dim()
    idx[ax] = sl
    return t[tuple(idx)]


def _up(v, nc, dim):
    t = v.reshape((dim + 1,) + tuple(reversed(nc)))
    for ax in range(1, dim + 1):
        even, odd = t, 0.5 * (_along(t, ax, slice(0, -1)) + _along(t, ax, slice(1, None)))
        shape = list(t.shape)
        shape[ax] = 2 * shape[ax] - 1
        t = torch.empty(shape, dtype=t.dtype, device=t.device)
        _along(t, ax, slice(0, None, 2)).copy_(even)
        _along(t, ax, slice(1, None, 2)).copy_(odd)
    return t.reshape(-1)


def _down(v, nf, dim, combine, scale):
    t = v.reshape((dim + 1,) + tuple(reversed(nf)))
    for ax in range(1, dim + 1):
        out, odd = _along(t, ax, slice(0, None, 2)).clone(), scale * _along(t, ax, slice(1, None, 2))
        left, right = _along(out, ax, slice(1, None)), _along(out, ax, slice(0, -1))
        left.copy_(combine(left, odd))
        right.copy_(combine(right, odd))
        t = out
    return t.reshape(-1)


def _network(flat, f):
    """The network in 64 bits from its FP32 parameters and input planes."""
    shapes = learned.layer_shapes()
    ws, off = [], 0
    for co, ci, k in shapes:
        w = flat[off:off + co * ci * k * k].reshape(co, ci, k, k)
        off += co * ci * k * k
        ws.append((w, flat[off:off + co]))
        off += co
    t, skips = f[None], []

    def conv(t, i):
        w, b = ws[i]
        return nnf.conv2d(t, w, b, padding=w.shape[-1] // 2)

    for k in range(4):
        if k:
            t = nnf.avg_pool2d(t, 2)
        t = torch.relu(conv(torch.relu(conv(t, 2 * k)), 2 * k + 1))
        skips.append(t)
    for d, k in enumerate((2, 1, 0)):
        t = torch.cat([t.repeat_interleave(2, 2).repeat_interleave(2, 3), skips[k]], 1)
        t = torch.relu(conv(torch.relu(conv(t, 8 + 2 * d)), 9 + 2 * d))
    return conv(t, 14)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None  # a whole solver
    s = prepare(case, seed)
    p = 5e-4
    if kind == "batch":
        hv, en = [], []
        for k, n in enumerate(_batch_shapes(case)):
            h = 1.0 / (max(n) - 1)
            F = _Functional(n, h, LS_OVER_H * h, p * (1 + k % 3))
            hv.append(F.hessvec(s["x"][k].double(), s["v"][k].double()))
            en.append(F.energy(s["x64"][k]))
        return {"hv": hv, "energy": en}
    n = _shape(case)
    dim, h = len(n), 1.0 / (max(n) - 1)
    F = _Functional(n, h, LS_OVER_H * h, p)
    if kind == "newton":
        return {"energy": F.energy(s["x"]), "gradient": F.gradient(s["x"]),
                "hv": [F.hessvec(s["x"], v) for v in s["v"]]}
    if kind == "product":
        return F.hessvec(s["x"].double(), s["v"].double())
    if kind == "stopping":
        return {"gradient": F.gradient(s["x"]), "energy": F.energy(s["x"])}
    if kind == "transfer":
        nc = [(v - 1) // 2 + 1 for v in n]
        add = lambda a, b: a + b  # noqa: E731
        ones = _down(torch.ones_like(s["x"]), n, dim, add, 0.5)
        return {"x": _down(s["x"], n, dim, add, 0.5) / ones, "g": _down(s["g"], n, dim, add, 0.5),
                "lo": _down(s["lo"], n, dim, torch.maximum, 1.0), "hi": _down(s["hi"], n, dim, torch.minimum, 1.0),
                "s": _up(s["sc"], nc, dim)}
    if kind == "galerkin":
        sizes = [[(v - 1) // (1 << l) + 1 for v in n] for l in reversed(range(case["levels"]))]
        out = []
        for l in range(len(sizes) - 1):
            v = s["v"][l].double()
            for k in range(l, len(sizes) - 1):
                v = _up(v, sizes[k], dim)
            v = F.hessvec(s["x"].double(), v)
            for k in reversed(range(l + 1, len(sizes))):
                v = _down(v, sizes[k], dim, lambda a, b: a + b, 0.5)
            out.append(v)
        return out
    L = s["L"]
    if kind == "propose":
        N, x, r = s["H"].nodes(), s["x"], s["p_new"] / s["p_prev"]
        f = torch.zeros((5, L.Hp, L.Wp), dtype=torch.float64, device="cuda")
        c = x[2 * N:].reshape(n[1], n[0])
        f[0, :n[1], :n[0]] = x[:N].reshape(n[1], n[0]) * (E_MOD / s["p_prev"])
        f[1, :n[1], :n[0]] = x[N:2 * N].reshape(n[1], n[0]) * (E_MOD / s["p_prev"])
        f[2, :n[1], :n[0]] = c
        f[3, :n[1], :n[0]] = r
        f[4, :n[1], :n[0]] = c - s["c_before"].reshape(n[1], n[0])
        flat = torch.from_numpy(_params(seed + 7, learned.layer_shapes())).cuda().double()
        y = _network(flat, f)
        yv = y[:, :n[1], :n[0]].reshape(3, -1)
        dp = s["p_new"] - s["p_prev"]
        xhat = torch.cat([r * x[:N] + dp / E_MOD * yv[0], r * x[N:2 * N] + dp / E_MOD * yv[1], x[2 * N:] + dp * yv[2]])
        return {"y": y, "xhat": xhat}
    flat = torch.from_numpy(s["flat"]).cuda().double().requires_grad_(True)
    ys, losses, grads = [], [], 0
    for f, t in s["data"]:
        y = _network(flat, f.double())
        loss = (0.5 * ((y - t.double()) * L.mask.double()) ** 2).sum() / (3 * L.n_valid)
        grads = grads + torch.autograd.grad(loss, flat)[0]
        ys.append(y.detach())
        losses.append(float(loss))
    return {"y": ys, "loss": losses, "grads": grads.cpu().numpy()}
