"""The calls whose time this repository looks after, over the range of sizes its users run.

A user of the solver opens a load increment, iterates it and reads the fields back; a user of
the learned warm start runs the network's forward pass once per increment and its training step
thousands of times before that.  Each case is one such call, through the package's public entry
points (``Grid``, ``Batch``, ``Net``).

Solver cases restore a device checkpoint, open one increment, iterate it a fixed number of
times (``max_iter``), commit the iterate and copy the fields to pinned host memory.  A solve to
tolerance is the same call with more iterations (13,100 to 45,900 per localizing increment of
the 64 x 64 box, 13,000 for the 511^3 one); the count is fixed here so that every pass does the
same work.  The history is that of a box loaded close to yield: a pure-shear stress with smooth
variations, a weak inclusion, 1 % cohesion noise and smooth velocity perturbations, so that part
of the cells return to the yield surface in every pass.

``exact`` restates the method in plain torch, in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2305_01701_gb300 as P

DT = 1e-4          # load increment of the repository's configurations (rate 1)
K_BULK, G_SHEAR = 2.0, 1.0


# ---- the cases -------------------------------------------------------------------------------

def _solve(name, n, precision, iters, n_chk, **more):
    c = {"kind": "solve", "nx": n[0], "ny": n[1], "nz": n[2] if len(n) == 3 else 0, "precision": precision,
         "iters": iters, "n_chk": n_chk, "Lx": 1.0, "Ly": 1.0, "Lz": 1.0, "mu_s": 0.0, "jaumann": True,
         "incompressible": False, "cell_g": False, "body_force": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def _net(name, kind, size, base, samples, levels=3):
    c = {"kind": kind, "X": size[0], "Y": size[1], "Z": size[2] if len(size) == 3 else 0, "base": base,
         "samples": samples, "levels": levels}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest grid in use: the 64 x 64 FP64 box, where launches and latency count
        _solve("solve2d-fp64-64", (64, 64), "fp64", 500, 100),
        # the 511 x 511 visco-elasto-plastic FP64 box
        _solve("solve2d-fp64-511-maxwell", (511, 511), "fp64", 300, 100, mu_s=1e-3),
        # one 2D grid in FP32: the 2:1 box of the symmetry study, without the Jaumann term
        _solve("solve2d-fp32-383x191", (383, 191), "fp32", 500, 100, Lx=2.0, jaumann=False),
        # 256 uneven 2D grids in one persistent launch per sweep (after the autotuner)
        {"name": "batch2d-fp32-256", "kind": "batch", "count": 256, "precision": "fp32", "iters": 400, "n_chk": 200,
         "smallest": 127, "largest": 511},
        # a small ragged 3D box with unequal sides and a Maxwell viscosity
        _solve("solve3d-fp32-90x40x24-maxwell", (90, 40, 24), "fp32", 500, 100, Lx=2.0, Ly=1.0, Lz=0.5, mu_s=1e-3),
        # the 127^3 box
        _solve("solve3d-fp32-127", (127, 127, 127), "fp32", 400, 100),
        # a large box (the production range goes on to 511^3 with the same kernels)
        _solve("solve3d-fp32-383", (383, 383, 383), "fp32", 300, 100),
        # plain FP64 in 3D, the baseline that users check the mixed solve against
        _solve("solve3d-fp64-127", (127, 127, 127), "fp64", 100, 100),
        # the heterogeneous box: a shear modulus per cell
        _solve("solve3d-fp32-95-cell-g", (95, 95, 95), "fp32", 200, 100, cell_g=True),
        # the warm start's inference before each large 3D increment
        _net("net3d-forward-64", "forward", (64, 64, 64), 32, 1),
        # its gradients (a training step without the optimiser), two samples
        _net("net3d-gradients-64", "gradients", (64, 64, 64), 32, 2),
        # a training step of the 2D network
        _net("net2d-train-48", "train", (48, 48), 16, 8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve2d", "solve2d", "solve3d", "solve3d", "solve3d", "batch", "net", "net"])
    if kind == "solve2d":
        prec = rng.choice(["fp32", "fp64"])
        n = (_log(rng, 24, 1023 if prec == "fp32" else 511), _log(rng, 24, 1023 if prec == "fp32" else 511))
        chk = rng.choice([50, 100])
        return _solve(None, n, prec, chk * rng.choice([2, 3, 4]), chk, Lx=rng.choice([1.0, 2.0]),
                      mu_s=rng.choice([0.0, 0.0, 1e-3]), jaumann=rng.random() < 0.8,
                      incompressible=rng.random() < 0.15, cell_g=rng.random() < 0.15, body_force=rng.random() < 0.1)
    if kind == "solve3d":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        hi = 255 if prec == "fp32" else 127
        n = tuple(_log(rng, 16, hi) for _ in range(3))
        chk = rng.choice([50, 100])
        return _solve(None, n, prec, chk * rng.choice([1, 2]), chk, Lx=rng.choice([1.0, 2.0]), Lz=rng.choice([1.0, 0.5]),
                      mu_s=rng.choice([0.0, 0.0, 1e-3]), jaumann=rng.random() < 0.8,
                      incompressible=rng.random() < 0.15, cell_g=rng.random() < 0.15, body_force=rng.random() < 0.1)
    if kind == "batch":
        lo = _log(rng, 31, 255)
        return {"kind": "batch", "count": _log(rng, 2, 192), "precision": rng.choice(["fp32", "fp32", "fp64"]),
                "iters": rng.choice([100, 200]), "n_chk": rng.choice([50, 100]), "smallest": lo,
                "largest": rng.randrange(lo, 512)}
    kind = rng.choice(["forward", "forward_static", "gradients", "train"])
    levels = rng.choice([2, 3, 3])
    m = 1 << (levels - 1)
    base = rng.choice([16, 32])
    static = kind == "forward_static"      # its activations have to fit a fixed array
    base = 16 if static else base
    if rng.random() < 0.5:
        size = tuple(m * _log(rng, 16 // m, 128 // m) for _ in range(2))
        return _net(None, kind, size, base, rng.randrange(1, 3 if static else 9), levels)
    size = tuple(m * _log(rng, 8 // m, (32 if static else 48) // m) for _ in range(3))
    return _net(None, kind, size, base, 1 if static else rng.randrange(1, 3), levels)


# ---- inputs ------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFF)
    return g


def _uniform(gen, shape):
    return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)


def _smooth(gen, shape, terms=3):
    """A smooth field of order one: products of a few random-phase waves along each axis."""
    r = _uniform(gen, (terms, len(shape), 2)).cpu().numpy()
    out = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for t in range(terms):
        f = None
        for d, m in enumerate(shape):
            x = torch.linspace(0.0, 1.0, m, device="cuda", dtype=torch.float64) if m > 1 else torch.zeros(
                1, device="cuda", dtype=torch.float64)
            w = torch.cos(2.0 * math.pi * ((1 + t + 2 * r[t, d, 0]) * x + r[t, d, 1]))
            w = w.view([-1 if e == d else 1 for e in range(len(shape))])
            f = w if f is None else f * w
        out += f
    return out / terms


def _shape(n, stag):
    """C-order shape (x fastest) of a field staggered along the directions in ``stag``."""
    return tuple(n[d] + (1 if d in stag else 0) for d in reversed(range(len(n))))


def _pairs(nd):
    return [(0, 1)] if nd == 2 else [(0, 1), (0, 2), (1, 2)]


def _field_names(nd):
    if nd == 2:
        return ["vx", "vy", "txx", "tyy", "txy", "p", "epl"]
    return ["vx", "vy", "vz", "txx", "tyy", "tzz", "txy", "txz", "tyz", "p", "epl"]


def _rates(nd):
    return [1.0, -1.0] if nd == 2 else [1.0, 0.0, -1.0]


def _inside(a, dims):
    """A view of ``a`` without its first and last layer along the directions in ``dims``."""
    nd = a.dim()
    for d in dims:
        ax = nd - 1 - d
        a = a.narrow(ax, 1, a.shape[ax] - 2)
    return a


def _history(n, L, seed):
    """Cohesion (with a weak inclusion and 1 % noise), and the fields of a box loaded close to yield."""
    nd = len(n)
    gen = _gen(seed)
    cshape = _shape(n, ())
    axes = [(-0.5 * L[d] + (torch.arange(n[d], device="cuda", dtype=torch.float64) + 0.5) * (L[d] / n[d])) for d in range(nd)]
    c = 1.5e-3 * (1.0 + 0.01 * (2.0 * _uniform(gen, cshape) - 1.0))
    centre = (_uniform(gen, (nd,)).cpu().numpy() - 0.5) * 0.5
    r2 = torch.zeros(cshape, device="cuda", dtype=torch.float64)
    for d in range(nd):
        r2 += ((axes[d] - centre[d] * L[d]) ** 2).view([-1 if e == nd - 1 - d else 1 for e in range(nd)])
    c = torch.where(r2 <= (0.08 * min(L)) ** 2, 0.5 * c, c).contiguous()
    level = 1.07e-3 if nd == 2 else 1.56e-3
    f = {}
    rates = _rates(nd)
    m = 1.0 + 0.06 * _smooth(gen, cshape)
    for d in range(nd):
        f["t" + "xyz"[d] * 2] = rates[d] * level * m + 5e-6 * _smooth(gen, cshape)
    for a, b in _pairs(nd):
        e = torch.zeros(_shape(n, (a, b)), device="cuda", dtype=torch.float64)
        s = _smooth(gen, e.shape) + 0.2 * (2.0 * _uniform(gen, e.shape) - 1.0)
        _inside(e, (a, b)).copy_(3e-5 * _inside(s, (a, b)))   # free slip: no shear on the walls
        f["t" + "xyz"[a] + "xyz"[b]] = e
    f["p"] = 3e-5 * _smooth(gen, cshape)
    f["epl"] = 1e-3 * torch.clamp(0.6 + _smooth(gen, cshape), min=0.0)
    for d in range(nd):
        x = (-0.5 * L[d] + torch.arange(n[d] + 1, device="cuda", dtype=torch.float64) * (L[d] / n[d]))
        v = rates[d] * x.view([-1 if e == nd - 1 - d else 1 for e in range(nd)]).expand(_shape(n, (d,))).contiguous()
        _inside(v, (d,)).add_(0.01 * _inside(_smooth(gen, v.shape), (d,)))
        f["v" + "xyz"[d]] = v
    return c, f


def _cell_modulus(n, L):
    """The repository's heterogeneous shear modulus: 1 at the centre, 1.2 at the walls."""
    nd = len(n)
    r2 = torch.zeros(_shape(n, ()), device="cuda", dtype=torch.float64)
    for d in range(nd):
        x = -0.5 * L[d] + (torch.arange(n[d], device="cuda", dtype=torch.float64) + 0.5) * (L[d] / n[d])
        r2 += (x ** 2).view([-1 if e == nd - 1 - d else 1 for e in range(nd)])
    return 1.2 - 0.2 * torch.exp(-r2 / (0.2 * min(L)) ** 2)


def _body_force(n):
    """A weight along y (faces), as host arrays."""
    nd = len(n)
    return [np.full(_shape(n, (d,)), -1e-4 if d == 1 else 0.0) for d in range(nd)]


class _Box:
    """One grid with its material, options and checkpoint, and the pinned buffers its fields are read into."""

    def __init__(self, n, L, precision, seed, case, phi=30.0, buffers=None):
        self.n, self.nd = n, len(n)
        c, f = _history(n, L, seed)
        self.names = _field_names(self.nd)
        self.g = g = P.Grid(self.nd, n, L, precision=P.FP64 if precision == "fp64" else P.FP32_MIXED)
        mu = case.get("mu_s", 0.0)
        g.set_material(K_BULK, G_SHEAR, mu if mu else math.inf, phi, 0.0, c.cpu().numpy())
        if case.get("cell_g"):
            g.set_shear_modulus(_cell_modulus(n, L).cpu().numpy())
        g.set_solver(tol=1e-10 if precision == "fp64" else 1e-7, max_iter=case["iters"], n_chk=case["n_chk"],
                     jaumann=case.get("jaumann", True), incompressible=case.get("incompressible", False))
        self.out = buffers or {k: torch.empty(tuple(f[k].shape), dtype=torch.float64, pin_memory=True) for k in self.names}
        for k in self.names:
            self.out[k].copy_(f[k])
            g.set_from(k, self.out[k].data_ptr(), f[k].numel())
        self.force = _body_force(n) if case.get("body_force") else None
        g.snapshot()

    def read(self):
        for k in self.names:
            self.g.get_into(k, self.out[k].data_ptr(), self.out[k].numel())
        return self.out


def _dims(case):
    n = (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())
    return n, (case["Lx"], case["Ly"], case["Lz"])[:len(n)]


def _batch_members(case, seed):
    """Sizes and friction angles of a batch's grids (square grids, sizes spread over the range)."""
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    lo, hi = case["smallest"], case["largest"]
    steps = [lo + (hi - lo) * q // 3 for q in range(4)]
    order = np.random.RandomState(case["count"]).randint(0, 4, case["count"])   # the sizes are the case's, not the seed's
    return [(int(steps[q]), 20.0 + 15.0 * float(r.rand())) for q in order]


class _BatchState:
    def __init__(self, case, seed):
        members = _batch_members(case, seed)
        total = {k: 0 for k in _field_names(2)}
        shapes = []
        for m, _ in members:
            s = {k: _shape((m, m), (0,) if k == "vx" else (1,) if k == "vy" else (0, 1) if k == "txy" else ()) for k in total}
            shapes.append(s)
            for k in total:
                total[k] += s[k][0] * s[k][1]
        self.out = {k: torch.empty(total[k], dtype=torch.float64, pin_memory=True) for k in total}
        at = {k: 0 for k in total}
        self.boxes = []
        for q, (m, phi) in enumerate(members):
            views = {}
            for k in total:
                cnt = shapes[q][k][0] * shapes[q][k][1]
                views[k] = self.out[k][at[k]:at[k] + cnt].view(shapes[q][k])
                at[k] += cnt
            self.boxes.append(_Box((m, m), (1.0, 1.0), case["precision"], seed + 7919 * q, case, phi, views))
        self.batch = P.Batch([b.g for b in self.boxes])
        self.batch.apply_increment(1.0, DT)
        self.batch.autotune()


class _NetState:
    def __init__(self, case, seed):
        nd = 3 if case["Z"] else 2
        self.size = [case["X"], case["Y"]] + ([case["Z"]] if nd == 3 else [])
        self.N = case["samples"]
        self.net = P.Net(nd, P.warm_in(nd), P.warm_out(nd), base=case["base"], levels=case["levels"])
        gen = _gen(seed)
        self.net.set_params(_net_params(case, nd, gen).cpu().numpy())
        self.x, self.t = _net_samples(case, nd, gen)
        self.y = torch.empty_like(self.t)
        torch.cuda.synchronize()


def _net_layers(case, nd):
    """(input channels, output channels, kernel size) of every convolution, in parameter order."""
    base, L, c, out = case["base"], case["levels"], P.warm_in(nd), []
    for lv in range(L):
        out += [(c, base << lv, 3), (base << lv, base << lv, 3)]
        c = base << lv
    for lv in range(L - 2, -1, -1):
        out += [((base << (lv + 1)) + (base << lv), base << lv, 3), (base << lv, base << lv, 3)]
    return out + [(base, P.warm_out(nd), 1)]


def _net_params(case, nd, gen):
    """Weights and biases of a network after some training: He-sized weights, small biases, a head
    that is no longer zero."""
    p = []
    for ci, co, k in _net_layers(case, nd):
        w = math.sqrt(2.0 / (ci * k ** nd)) if k == 3 else 0.2
        p.append(w * torch.randn(ci * co * k ** nd, generator=gen, device="cuda"))
        p.append(0.05 * torch.randn(co, generator=gen, device="cuda"))
    return torch.cat(p)


def _net_samples(case, nd, gen):
    """Features (smooth velocity change, stress and pressure over the cohesion; sparse plastic
    channels) and targets, per sample."""
    dims = [case["Z"], case["Y"], case["X"]] if nd == 3 else [case["Y"], case["X"]]
    cin, cout, N = P.warm_in(nd), P.warm_out(nd), case["samples"]
    x = 0.5 * torch.randn([N, cin] + dims, generator=gen, device="cuda")
    x += torch.randn([N, cin] + [1] * nd, generator=gen, device="cuda")
    x[:, -3] = torch.clamp(x[:, -3], min=0.0)
    x[:, -1] = torch.clamp(x[:, -1], min=0.0)
    t = torch.randn([N, cout] + dims, generator=gen, device="cuda")
    return x.contiguous(), t.contiguous()


def prepare(case, seed):
    if case["kind"] == "solve":
        n, L = _dims(case)
        return ("solve", _Box(n, L, case["precision"], seed, case))
    if case["kind"] == "batch":
        return ("batch", _BatchState(case, seed))
    return (case["kind"], _NetState(case, seed))


# ---- one pass ----------------------------------------------------------------------------------

def run(state):
    kind, s = state
    if kind == "solve":
        g = s.g
        g.restore()
        g.apply_increment(1.0, DT, P.LOAD_XY if s.nd == 2 else P.LOAD_XZ, s.force)
        g.solve_increment(raise_on_fail=False)
        g.commit_increment()
        return s.read()
    if kind == "batch":
        for b in s.boxes:
            b.g.restore()
        s.batch.apply_increment(1.0, DT)
        s.batch.solve_increment(raise_on_fail=False)
        for b in s.boxes:
            b.g.commit_increment()
            b.read()
        return s.out
    if kind == "forward":
        s.net.forward(s.x.data_ptr(), s.N, s.size, s.y.data_ptr())
        return s.y
    if kind == "forward_static":
        s.net.forward_static(s.x.data_ptr(), s.N, s.size, s.y.data_ptr())
        return s.y
    if kind == "gradients":
        loss, g = s.net.gradients(s.x.data_ptr(), s.t.data_ptr(), s.N, s.size)
        return {"loss": loss, "gradient": g}
    loss = s.net.train_step(s.x.data_ptr(), s.t.data_ptr(), s.N, s.size, 1e-3)
    return {"loss": loss, "params": s.net.get_params()}


# ---- what a pass cannot do without ----------------------------------------------------------------

# floating-point operations of one iteration per cell, counted from the method's formulas with
# every mean formed once
_FLOPS = {2: 90.0, 3: 220.0}


def _sweep_work(n, size, iters):
    nd, cells = len(n), float(np.prod(n))
    words = 19 if nd == 2 else 33     # fields one iteration reads and writes, each once
    return (iters + 1) * words * size * cells, (iters + 1) * _FLOPS[nd] * cells


def _net_macs(case):
    """Multiply-adds of the forward pass and of its first layer, parameters, and values of the
    input and output."""
    nd = 3 if case["Z"] else 2
    vox = case["samples"] * case["X"] * case["Y"] * (case["Z"] or 1)
    L = case["levels"]
    lv_of = [lv for lv in range(L) for _ in range(2)] + [lv for lv in range(L - 2, -1, -1) for _ in range(2)] + [0]
    macs = [ci * co * k ** nd * vox / (2 ** nd) ** lv for (ci, co, k), lv in zip(_net_layers(case, nd), lv_of)]
    par = sum(ci * co * k ** nd for ci, co, k in _net_layers(case, nd))
    return sum(macs), macs[0], par, vox * P.warm_in(nd), vox * P.warm_out(nd)


def work(case):
    if case["kind"] == "solve":
        n, _ = _dims(case)
        size = 8 if case["precision"] == "fp64" else 4
        b, f = _sweep_work(n, size, case["iters"])
        out = len(_field_names(len(n))) * 8.0 * float(np.prod(n))
        return {"bytes": b + 2 * out, "flops": f}
    if case["kind"] == "batch":
        b = f = 0.0
        for m, _ in _batch_members(case, 0):
            x, y = _sweep_work((m, m), 8 if case["precision"] == "fp64" else 4, case["iters"])
            b, f = b + x + 2 * 7 * 8.0 * m * m, f + y
        return {"bytes": b, "flops": f}
    macs, first, par, xin, xout = _net_macs(case)
    if case["kind"] in ("forward", "forward_static"):
        return {"bytes": 4 * (xin + xout) + 2 * par, "flops": 2 * macs}
    # the backward pass: the weights' gradients, and the inputs' of all layers but the first
    opt = 4 * 6 * par if case["kind"] == "train" else 4 * par
    return {"bytes": 4 * (xin + xout) + 2 * par + opt, "flops": 2 * (3 * macs - first)}


def tolerance(case):
    if case["kind"] in ("solve", "batch"):
        # seen between the sweep kernels and against exact(), with their sums in other orders:
        # 2e-13 in 64 bits, 6e-5 (v_y, the smallest velocity) to 1.2e-4 (shear) in 32, and in 32
        # single cells that one order returns to the yield surface and the other does not: their
        # plastic strain then differs by a whole increment's (1.3e-3 of the field, once its size)
        if case["precision"] == "fp64":
            return {"rel": 1e-11, "max": 1e-9}
        return {"rel": 5e-3, "max": 0.99}
    if case["kind"] in ("forward", "forward_static"):
        # BF16 inputs of the convolutions: 4e-3 to 7e-3 against exact()
        return {"rel": 1e-2, "max": 1e-1}
    if case["kind"] == "gradients":
        # 32-bit sums over all voxels: 1e-5 against exact()
        return {"rel": 4e-5, "max": 2e-3}
    # Adam divides by the gradient's own size: where a gradient is all rounding, its sign and the
    # weight's whole step are
    return {"rel": 1e-3, "max": 3e-1}


# ---- the same in plain torch, in 64 bits ------------------------------------------------------------

def _ax(a, d):
    return a.dim() - 1 - d


def _diff(a, d):
    ax = _ax(a, d)
    m = a.shape[ax]
    return a.narrow(ax, 1, m - 1) - a.narrow(ax, 0, m - 1)


def _avg(a, d):
    ax = _ax(a, d)
    m = a.shape[ax]
    return 0.5 * (a.narrow(ax, 1, m - 1) + a.narrow(ax, 0, m - 1))


def _pad(a, dims):
    """Zero layers on both sides along the directions in ``dims``."""
    p = []
    for d in range(a.dim()):       # torch pads from the last axis (x) on
        p += [1, 1] if d in dims else [0, 0]
    return torch.nn.functional.pad(a, p)


def _edge_mean(Gc, a, b):
    """The mean of a centre field at the edges of the pair (a, b), indices clamped at the walls."""
    for d in (a, b):
        ax = _ax(Gc, d)
        m = Gc.shape[ax]
        Gc = torch.cat([Gc.narrow(ax, 0, 1), Gc, Gc.narrow(ax, m - 1, 1)], ax)
        Gc = _avg(Gc, d)
    return Gc


def _solve_exact(n, L, case, seed, phi=30.0):
    nd = len(n)
    c, f = _history(n, L, seed)
    h = [L[d] / n[d] for d in range(nd)]
    pairs = _pairs(nd)
    mu = case.get("mu_s", 0.0) or math.inf
    Gc = _cell_modulus(n, L) if case.get("cell_g") else torch.full_like(c, G_SHEAR)
    Gm = float(Gc.max())

    def eta_of(G):
        return G * DT if math.isinf(mu) else 1.0 / (1.0 / (G * DT) + 1.0 / mu)

    eta = eta_of(Gm)
    Re, Vp = 3.0 * math.sqrt(10.0) * math.pi / 2.0, 0.9 / math.sqrt(nd) * min(h)
    rho = Re * eta / (Vp * max(L))
    Gt = rho * Vp * Vp / (0.5 + 4.0 / 3.0)
    Kt = 0.5 * Gt
    bt = (1.0 / (2.0 * Gt)) / (1.0 / (2.0 * Gt) + 1.0 / (2.0 * eta))
    inc = case.get("incompressible", False)
    bp = 1.0 if inc else (1.0 / Kt) / (1.0 / Kt + 1.0 / (K_BULK * DT))
    ph = math.radians(phi)
    if nd == 2:
        A, B = math.sin(ph), math.cos(ph)
    else:
        A = 6.0 * math.sin(ph) / (math.sqrt(3.0) * (3.0 - math.sin(ph)))
        B = 6.0 * math.cos(ph) / (math.sqrt(3.0) * (3.0 - math.sin(ph)))
    Yc = B * c
    te_c, c2_c = 2.0 * eta_of(Gc), eta_of(Gc) / (Gc * DT)
    te_e, c2_e = {}, {}
    for q in pairs:
        Ge = _edge_mean(Gc, *q)
        te_e[q], c2_e[q] = 2.0 * eta_of(Ge), eta_of(Ge) / (Ge * DT)
    wj = DT if case.get("jaumann", True) else 0.0
    old_n = [f["t" + "xyz"[d] * 2] for d in range(nd)]
    old_s = {q: f["t" + "xyz"[q[0]] + "xyz"[q[1]]] for q in pairs}
    rq = {q: wj * old_s[q] for q in pairs}
    rd = {q: wj * (old_n[q[1]] - old_n[q[0]]) for q in pairs}
    force = [torch.tensor(a, device="cuda") for a in _body_force(n)] if case.get("body_force") else None

    def mean4(a, q):
        return _avg(_avg(a, q[0]), q[1])

    def trial(v):
        es, om = {}, {}
        for a, b in pairs:
            x = _inside(_diff(v[a], b), (a,)) / h[b]
            y = _inside(_diff(v[b], a), (b,)) / h[a]
            es[a, b], om[a, b] = _pad(0.5 * (x + y), (a, b)), _pad(0.5 * (x - y), (a, b))
        e = [_diff(v[d], d) / h[d] for d in range(nd)]
        div = sum(e)
        Pm = {q: mean4(rq[q] * om[q], q) for q in pairs}
        if nd == 2:
            rot = [2 * Pm[0, 1], -2 * Pm[0, 1]]
        else:
            xy, xz, yz = Pm[0, 1], Pm[0, 2], Pm[1, 2]
            rot = [2 * (xy + xz), -2 * (xy - yz), -2 * (xz + yz)]
        Tn = [c2_c * old_n[d] + te_c * (e[d] - div / 3.0) + c2_c * rot[d] for d in range(nd)]
        Ts = {}
        for q in pairs:
            w = _inside(om[q], q) * mean4(rd[q], q)
            if nd == 3:
                def at(m, src):
                    """Mean of the edge field ``src`` of the pair m at this pair's interior edges."""
                    g = src[m]
                    for d in m:
                        g = _avg(g, d) if d not in q else _inside(g, (d,))
                    for d in q:
                        if d not in m:
                            g = _avg(g, d)
                    return g
                if q == (0, 1):
                    w = w + at((1, 2), rq) * at((0, 2), om) + at((0, 2), rq) * at((1, 2), om)
                elif q == (0, 2):
                    w = w + at((1, 2), rq) * at((0, 1), om) - at((0, 1), rq) * at((1, 2), om)
                else:
                    w = w - at((0, 1), rq) * at((0, 2), om) - at((0, 2), rq) * at((0, 1), om)
            Ts[q] = _pad(_inside(c2_e[q] * old_s[q] + te_e[q] * es[q], q) + _inside(c2_e[q], q) * w, q)
        return Tn, Ts, div

    def ret(Tn, Ts, p):
        J2 = sum(mean4(Ts[q], q) ** 2 for q in pairs) + 0.5 * sum(t * t for t in Tn)
        sj = torch.sqrt(J2)
        Y = torch.clamp(A * p + Yc, min=0.0)
        s = torch.where(sj > Y, Y / sj, torch.ones_like(sj))
        return s, [s * t for t in Tn], {q: _pad(mean4(s, q) * _inside(Ts[q], q), q) for q in pairs}

    v = [f["v" + "xyz"[d]].clone() for d in range(nd)]    # the walls already move at the loading rate
    Tn, Ts, div = trial(v)
    p = f["p"].clone() if inc else f["p"] - K_BULK * DT * div
    s, tn, ts = ret(Tn, Ts, p)
    for k in range(case["iters"] + 1):
        Tn, Ts, div = trial(v)
        Rn = [bt * tn[d] + (1.0 - bt) * Tn[d] for d in range(nd)]
        Rs = {q: bt * ts[q] + (1.0 - bt) * Ts[q] for q in pairs}
        p = p - Kt * div if inc else bp * p + (1.0 - bp) * (f["p"] - K_BULK * DT * div)
        s, tn, ts = ret(Rn, Rs, p)
        if k == case["iters"]:
            break               # the iterate that is committed
        for d in range(nd):
            R = _diff(tn[d] - p, d) / h[d]
            for q in pairs:
                if d in q:
                    o = q[0] if d == q[1] else q[1]
                    R = R + _inside(_diff(ts[q], o), (d,)) / h[o]
            if force is not None:
                R = R + _inside(force[d], (d,))
            _inside(v[d], (d,)).add_(R / rho)
    dJ = sum(mean4(Ts[q] - ts[q], q) ** 2 for q in pairs) + 0.5 * sum((Tn[d] - tn[d]) ** 2 for d in range(nd))
    out = {"v" + "xyz"[d]: v[d] for d in range(nd)}
    out.update({"t" + "xyz"[d] * 2: tn[d] for d in range(nd)})
    out.update({"t" + "xyz"[a] + "xyz"[b]: ts[a, b] for a, b in pairs})
    out["p"] = p
    # in 32 bits a cell at the yield surface adds a whole increment's plastic strain or none
    out["epl"] = None if case["precision"] == "fp32" else \
        f["epl"] + torch.where(s < 1.0, DT * torch.sqrt(dJ) / te_c, torch.zeros_like(dJ))
    return out


def _net_exact(case, seed, grad):
    """The network on its BF16 weights (FP32 biases) and unrounded activations."""
    nd = 3 if case["Z"] else 2
    gen = _gen(seed)
    params = _net_params(case, nd, gen)
    x, t = _net_samples(case, nd, gen)
    x, t = x.double(), t.double()
    conv = torch.nn.functional.conv3d if nd == 3 else torch.nn.functional.conv2d
    pool = torch.nn.functional.avg_pool3d if nd == 3 else torch.nn.functional.avg_pool2d
    leaves, at = [], [0]

    def layer(a, ci, co, k):
        m = ci * co * k ** nd
        w = params[at[0]:at[0] + m].bfloat16().double().view([co, ci] + [k] * nd).requires_grad_(grad)
        b = params[at[0] + m:at[0] + m + co].double().requires_grad_(grad)
        at[0] += m + co
        leaves.extend([w, b])
        return conv(a, w, b, padding=k // 2)

    base, levels, skips = case["base"], case["levels"], []
    with torch.set_grad_enabled(grad):
        a, ci = x, P.warm_in(nd)
        for lv in range(levels):
            o = base << lv
            a = torch.relu(layer(a, ci, o, 3))
            a = torch.relu(layer(a, o, o, 3))
            ci = o
            if lv < levels - 1:
                skips.append(a)
                a = pool(a, 2)
        for lv in range(levels - 2, -1, -1):
            o, up = base << lv, base << (lv + 1)
            a = torch.nn.functional.interpolate(a, scale_factor=2, mode="nearest")
            a = torch.relu(layer(torch.cat([a, skips[lv]], 1), up + o, o, 3))
            a = torch.relu(layer(a, o, o, 3))
        y = layer(a, base, P.warm_out(nd), 1)
        if not grad:
            return y, None, None
        loss = ((y - t) ** 2).mean()
        loss.backward()
    return y, float(loss.detach()), torch.cat([q.grad.reshape(-1) for q in leaves])


def exact(case, seed):
    if case["kind"] == "solve":
        n, L = _dims(case)
        if float(np.prod(n)) * case["iters"] > 1.2e9:
            return None     # minutes in plain torch
        return _solve_exact(n, L, case, seed)
    if case["kind"] == "batch":
        members = _batch_members(case, seed)
        if len(members) * case["iters"] > 8000:
            return None
        outs = [_solve_exact((m, m), (1.0, 1.0), case, seed + 7919 * q, phi) for q, (m, phi) in enumerate(members)]
        return {k: None if outs[0][k] is None else torch.cat([o[k].reshape(-1) for o in outs]) for k in outs[0]}
    if case["kind"] in ("forward", "forward_static"):
        return _net_exact(case, seed, False)[0]
    _, loss, g = _net_exact(case, seed, True)
    if case["kind"] == "gradients":
        return {"loss": loss, "gradient": g}
    # Adam's first step moves every weight by the learning rate's length whatever the size of its
    # gradient, so the updated weights say nothing about precision; the gradients case does
    return {"loss": loss, "params": None}
