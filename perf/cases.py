"""The workloads by which this library's speed is judged.

Each case is one call (or the few calls) that a program using the library makes
through the package's public classes, at the sizes of the repository's own
configurations, tests and benchmark:

* a whole solve to 1e-10: a small circle in FP64, the unit sphere at
  dx = 1/256 in mixed precision, a batch of ellipsoids with several right-hand
  sides, and a cold solve that builds its band and hierarchy first;
* the pieces a solve, a Krylov method or a time stepper calls on their own: the
  operator, smoothing sweeps, V-cycles and the outer residual;
* the learned smoother's network, forward (inference) and backward (training).

``exact`` evaluates the same quantities in 64 bits with plain torch: its own
closest points, band, stencils and multigrid.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1307_4354_gb300 as cpm

FP = {"f64": torch.float64, "f32": torch.float32}


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # The smallest whole problem: Fourier data on the unit circle, FP64 throughout,
        # 2 + 2 sweeps of omega = 2/3 down to dx = 1/8.  Latency of a complete solve.
        dict(name="circle_solve_f64", op="solve", surface="circle", p0=1.0, p1=0.0, p2=0.0, inv_dx=64,
             coarsest=8, mode="f64", nu=2, omega=2.0 / 3.0, inner=1, form="mbr"),
        # One application of the paper-form operator (Eq. 3.3) at the finest spacing of
        # Table 3.1: the matvec of a Krylov method or an explicit step on a curve.
        dict(name="circle_apply_paper_f64", op="apply", surface="circle", p0=1.0, p1=0.0, p2=0.0,
             inv_dx=640, prec="f64", form="paper"),
        # One FP64 matvec M u on an ellipsoid at a spacing of the batched workload.
        dict(name="ellipsoid_apply_f64", op="apply", surface="ellipsoid", p0=1.1, p1=0.8, p2=0.7,
             inv_dx=96, prec="f64", form="mbr"),
        # Four weighted Jacobi sweeps on the finest level of the headline problem, FP32: the
        # step that a mixed-precision solve spends most of its time in.
        dict(name="sphere_smooth_f32", op="smooth", surface="sphere", p0=1.0, p1=0.0, p2=0.0, inv_dx=256,
             prec="f32", form="mbr", sweeps=4, omega=0.8),
        # One FP32 V-cycle from zero, the preconditioner of an outer iteration.
        dict(name="sphere_vcycle_f32", op="vcycle", surface="sphere", p0=1.0, p1=0.0, p2=0.0, inv_dx=128,
             coarsest=8, prec="f32", form="mbr", nu=4, omega=0.8, residual="plain"),
        # One FP64 V-cycle on a torus with the library's default options; its coarsest level
        # (dx = 1/12, 23 thousand points) is above the size limit of the FP64 inverse.
        dict(name="torus_vcycle_f64", op="vcycle", surface="torus", p0=1.0, p1=0.5, p2=0.0, inv_dx=96,
             coarsest=12, prec="f64", form="mbr", nu=3, omega=0.8, residual="extended"),
        # The outer residual of a fine torus: what every outer iteration ends with.
        dict(name="torus_residual", op="residual", surface="torus", p0=1.0, p1=0.4, p2=0.0, inv_dx=256),
        # The headline: unit sphere, dx = 1/256, mixed precision to 1e-10.
        dict(name="sphere_solve_mixed", op="solve", surface="sphere", p0=1.0, p1=0.0, p2=0.0, inv_dx=256,
             coarsest=8, mode="mixed", nu=4, omega=0.8, inner=3, form="mbr"),
        # Four ellipsoids of uneven band sizes with four right-hand sides each, solved as one
        # batch in mixed precision.
        dict(name="batch_solve_mixed", op="batch", surfaces=4, surface_seed=1, axis_lo=0.8, axis_hi=1.2,
             n_rhs=4, nu=4, omega=0.8, inner=2),
        # A new surface, solved once: band, hierarchy, one mixed-precision solve.
        dict(name="sphere_cold_solve", op="cold", surface="sphere", p0=1.0, p1=0.0, p2=0.0, inv_dx=64,
             coarsest=8, mode="mixed", nu=4, omega=0.8, inner=2, form="mbr"),
        # Inference of the learned smoother on the torus that it is evaluated on.
        dict(name="smoother_forward", op="mlp", surface="torus", p0=1.0, p1=0.35, p2=0.0, inv_dx=128),
        # Loss and gradient of one training field of the learned smoother.
        dict(name="smoother_backward", op="mlp_grad", surface="ellipsoid", p0=1.05, p1=0.9, p2=0.75,
             inv_dx=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_surface(rng, lo, hi):
    """A surface of the kinds in use and 1/dx in [lo, hi], odd sizes among them."""
    kind = rng.choice(["sphere", "torus", "ellipsoid"])
    if kind == "sphere":
        p = (rng.uniform(0.8, 1.2), 0.0, 0.0)
    elif kind == "torus":
        p = (rng.uniform(0.95, 1.2), rng.uniform(0.35, 0.5), 0.0)
    else:
        p = tuple(rng.uniform(0.7, 1.15) for _ in range(3))
    # 4/dx whole; at most as many points as the unit sphere at 1/hi
    area = {"sphere": 12.57 * p[0] ** 2, "torus": 39.48 * p[0] * p[1], "ellipsoid": 12.57}[kind]
    inv_dx = min(_log_int(rng, lo, hi), int(hi * math.sqrt(12.57 / max(area, 12.57))))
    return dict(surface=kind, p0=round(p[0], 4), p1=round(p[1], 4), p2=round(p[2], 4), inv_dx=inv_dx)


def draw(rng):
    op = rng.choice(["circle_solve", "circle_apply", "apply", "smooth", "vcycle", "vcycle", "residual",
                     "solve", "solve", "batch", "mlp", "mlp_grad"])
    if op == "circle_solve":
        q, k = rng.randint(7, 13), rng.randint(2, 6)
        return dict(op="solve", surface="circle", p0=1.0, p1=0.0, p2=0.0, inv_dx=q << k, coarsest=q,
                    mode=rng.choice(["f64", "mixed"]), nu=rng.choice([3, 4]), omega=0.8, inner=1,
                    form="mbr")
    if op == "circle_apply":
        return dict(op="apply", surface="circle", p0=round(rng.uniform(0.8, 1.2), 4), p1=0.0, p2=0.0,
                    inv_dx=_log_int(rng, 40, 1000), prec=rng.choice(["f64", "f32"]),
                    form=rng.choice(["mbr", "paper"]))
    if op == "apply":
        return dict(op="apply", **_draw_surface(rng, 32, 256), prec=rng.choice(["f64", "f32"]),
                    form=rng.choice(["mbr", "mbr", "paper"]))
    if op == "smooth":
        return dict(op="smooth", **_draw_surface(rng, 32, 256), prec=rng.choice(["f64", "f32", "f32"]),
                    form=rng.choice(["mbr", "mbr", "paper"]), sweeps=rng.randint(1, 4), omega=0.8)
    if op == "residual":
        return dict(op="residual", **_draw_surface(rng, 32, 256))
    if op in ("mlp", "mlp_grad"):
        return dict(op=op, **_draw_surface(rng, 32, 200 if op == "mlp" else 96))
    if op == "batch":
        return dict(op="batch", surfaces=rng.randint(2, 4), surface_seed=rng.randint(2, 1 << 20),
                    axis_lo=0.85, axis_hi=1.15, n_rhs=rng.randint(1, 5), nu=rng.choice([3, 4]), omega=0.8,
                    inner=2)
    # whole cycles and solves on spheres and tori with a nested hierarchy
    if rng.random() < 0.7:
        q, surf = rng.choice([6, 7, 8]), dict(surface="sphere", p0=1.0, p1=0.0, p2=0.0)
        k = rng.randint(1, 5 if q < 8 else 4)
    else:
        q, surf = rng.choice([11, 12, 13]), dict(surface="torus", p0=1.0, p1=0.5, p2=0.0)
        k = rng.randint(1, 3)
    base = dict(surf, inv_dx=q << k, coarsest=q, form="mbr", nu=rng.choice([3, 4]), omega=0.8)
    if op == "vcycle":
        return dict(base, op="vcycle", prec=rng.choice(["f64", "f32"]),
                    residual=rng.choice(["plain", "extended"]))
    mode = rng.choice(["mixed", "mixed", "f64"])
    return dict(base, op="solve", mode=mode, inner=rng.randint(1, 3) if mode == "mixed" else 1)


# ----------------------------------------------------------------- inputs
def _params(case):
    n = {"circle": 1, "sphere": 1, "torus": 2, "ellipsoid": 3}[case["surface"]]
    return tuple(case["p%d" % i] for i in range(n))


def _ellipsoids(case):
    """[(semi-axes, 1/dx)] of a batch."""
    rng = np.random.default_rng(case["surface_seed"])
    axes = rng.uniform(case["axis_lo"], case["axis_hi"], size=(case["surfaces"], 3))
    pick = rng.integers(0, 3, size=case["surfaces"])
    return [(tuple(float(v) for v in axes[i]), (64, 96, 128)[pick[i]]) for i in range(case["surfaces"])]


def _field(y, seed):
    """A smooth field at points y of the surface: eight products of sines, wave
    numbers up to 4, random phases and amplitudes."""
    rng = np.random.default_rng(seed)
    d = y.shape[1]
    out = torch.zeros(y.shape[0], dtype=torch.float64, device=y.device)
    for _ in range(8):
        k = rng.integers(-4, 5, size=d)
        ph = rng.uniform(0.0, 2 * math.pi, size=d)
        t = torch.full_like(out, float(rng.normal()))
        for a in range(d):
            t = t * torch.sin(float(k[a]) * y[:, a] + float(ph[a]))
        out += t
    return out


def _noise(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * 2 - 1


def _variable_c(y):
    return 1.0 + 0.5 * torch.sin(2 * math.pi * y[:, -1])


def _rhs(y, seed):
    return _field(y, seed) + _field(y * 0.5, seed + 1)


def _iterate(y, seed):
    """A vector as the cycles meet it: a smooth part and a rough one."""
    return 0.05 * _field(y, seed) + 0.002 * _noise(y.shape[0], seed + 7)


def _residual_like(y, seed):
    """A V-cycle's residual: oscillatory, largest value 1."""
    r = _field(y, seed) * (1 + 0.3 * _field(y * 3, seed + 5)) + 0.1 * _noise(y.shape[0], seed + 9)
    return r / r.abs().max()


def _network(seed):
    """He-scaled weights of the 31 -> 64 -> 64 -> 1 network with small biases."""
    rng = np.random.default_rng(seed)
    w1 = rng.standard_normal((32, 64)) * math.sqrt(2 / 31)
    w1[31] = 0.0
    parts = [w1, 0.1 * rng.standard_normal(64), rng.standard_normal((64, 64)) * math.sqrt(2 / 64),
             0.1 * rng.standard_normal(64), rng.standard_normal(64) * math.sqrt(2 / 64),
             0.1 * rng.standard_normal(1)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _points(band):
    """Closest points of B on the device."""
    _, cp, _ = band.export()
    return torch.from_numpy(cp[: band.nb]).cuda()


def _hierarchy(case, band, c=None):
    """The hierarchy that a program using this case's call keeps."""
    if case["op"] in ("solve", "cold", "vcycle"):
        return cpm.Hierarchy(band, coarsest_dx=1.0 / case["coarsest"], nu1=case["nu"], nu2=case["nu"],
                             omega=case["omega"], residual=case.get("residual", "plain"),
                             op_form=case["form"])
    # operator and smoother calls on one level: no coarser levels, no coarsest inverse
    return cpm.Hierarchy(band, coarsest_dx=1.0 / case["inv_dx"], coarse_sweeps=1,
                         omega=case.get("omega", 0.8), op_form=case.get("form", "mbr"), c_device=c)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        hs, fs = [], []
        for i, (axes, inv_dx) in enumerate(_ellipsoids(case)):
            band = cpm.Band("ellipsoid", axes, 1.0 / inv_dx)
            hs.append(cpm.Hierarchy(band, nu1=case["nu"], nu2=case["nu"], omega=case["omega"],
                                    residual="plain", coarse_f64_max=4096))
            y = _points(band)
            fs += [_rhs(y, 1000 * seed + 100 * i + 10 * k) for k in range(case["n_rhs"])]
        return dict(op=op, case=case, B=cpm.Batch(hs, case["n_rhs"]), f=fs)
    band = cpm.Band(case["surface"], _params(case), 1.0 / case["inv_dx"])
    y = _points(band)
    st = dict(op=op, case=case, band=band)
    if op in ("mlp", "mlp_grad"):
        st["H"] = _hierarchy(case, band, _variable_c(y))
        st["net"] = cpm.Smoother(params=_network(seed))
        st["H"].set_smoother(st["net"])
        st["r"] = _residual_like(y, seed).float()
        return st
    if op in ("solve", "cold"):
        st["f"] = _rhs(y, seed)
        if op == "solve":
            st["H"] = _hierarchy(case, band)
        else:
            band.close()
            del st["band"]
        return st
    st["H"] = _hierarchy(case, band)
    dt = FP[case.get("prec", "f64")]
    if op == "apply":
        st["u"] = _iterate(y, seed).to(dt)
    elif op == "residual":
        st["u"], st["f"] = _iterate(y, seed), _rhs(y, seed)
    else:
        st["f"] = _residual_like(y, seed).to(dt)
        st["u"] = (1e-3 * _iterate(y, seed)).to(dt) if op == "smooth" else torch.zeros_like(st["f"])
    return st


def run(st):
    op, case = st["op"], st["case"]
    if op == "apply":
        return st["H"].apply(st["u"])
    if op == "smooth":
        return st["H"].smooth(st["f"], st["u"], sweeps=case["sweeps"])
    if op == "vcycle":
        st["u"].zero_()
        return st["H"].vcycle(st["f"], st["u"])
    if op == "residual":
        return st["H"].residual(st["f"], st["u"])
    if op == "solve":
        return st["H"].solve(st["f"], mode=case["mode"], inner_cycles=case["inner"])[0]
    if op == "cold":
        band = cpm.Band(case["surface"], _params(case), 1.0 / case["inv_dx"])
        H = _hierarchy(case, band)
        u, _ = H.solve(st["f"], mode=case["mode"], inner_cycles=case["inner"])
        H.close()
        band.close()
        return u
    if op == "batch":
        return st["B"].solve(st["f"], mode="mixed", inner_cycles=case["inner"])[0]
    if op == "mlp":
        return st["H"].smoother_correction(st["r"])
    return list(st["H"].smoother_loss_grad(st["r"]))


# ----------------------------------------------------------------- work
def _sizes(kind, params, inv_dx):
    """(|B|, |B+|) from the surface's measure and the band's thickness."""
    if kind == "circle":
        n = 2 * math.pi * params[0] * 2 * math.sqrt(13.0) * inv_dx
        return n, n * (1 + 1 / math.sqrt(13.0))
    if kind == "ellipsoid":
        e = 1.6075
        a, b, c = (v ** e for v in params)
        area = 4 * math.pi * ((a * b + a * c + b * c) / 3) ** (1 / e)
    else:
        area = 4 * math.pi * params[0] ** 2 if kind == "sphere" else 4 * math.pi ** 2 * params[0] * params[1]
    n = area * 2 * math.sqrt(17.0) * inv_dx ** 2
    return n, n * 1.2


def _sweep(nb, npl, b, d):
    """One Jacobi sweep or residual: u, f and the diagonal read, one result written,
    d fractions per point of B+ read; the separable contraction and the stencil."""
    return np.array([4 * b * nb + d * b * npl, npl * 2 * sum(4 ** k for k in range(1, d + 1)) + nb * (4 * d + 6)])


def _cycle(case, kind, params, inv_dx, coarsest, b, nu):
    d = 2 if kind == "circle" else 3
    w = np.zeros(2)
    while True:
        nb, npl = _sizes(kind, params, inv_dx)
        if inv_dx // 2 < coarsest or inv_dx % 2:
            # the direct solve, counted as one pass over its right-hand side and result
            return w + np.array([2 * b * nb, 2 * nb])
        w += (2 * nu + 1) * _sweep(nb, npl, b, d) + np.array([2 * b * nb, 4.0 * (2 ** d) * nb])
        inv_dx //= 2


def work(case):
    op = case["op"]
    if op == "batch":
        w = np.zeros(2)
        for axes, inv_dx in _ellipsoids(case):
            nb, npl = _sizes("ellipsoid", axes, inv_dx)
            one = case["inner"] * _cycle(case, "ellipsoid", axes, inv_dx, 12, 4, case["nu"])
            w += case["n_rhs"] * 4 * (one + _sweep(nb, npl, 8, 3))
        return dict(bytes=float(w[0]), flops=float(w[1]))
    kind, params, inv_dx = case["surface"], _params(case), case["inv_dx"]
    nb, npl = _sizes(kind, params, inv_dx)
    d = 2 if kind == "circle" else 3
    b = 4 if case.get("prec") == "f32" else 8
    if op in ("solve", "cold"):
        outer = 13 if case["mode"] == "f64" else {1: 12, 2: 6}.get(case["inner"], 4)
        cb = 8 if case["mode"] == "f64" else 4
        w = outer * (case["inner"] * _cycle(case, kind, params, inv_dx, case["coarsest"], cb, case["nu"])
                     + _sweep(nb, npl, 8, d))
    elif op == "vcycle":
        w = _cycle(case, kind, params, inv_dx, case["coarsest"], b, case["nu"])
    elif op == "smooth":
        w = case["sweeps"] * _sweep(nb, npl, b, d)
    elif op == "residual":
        w = _sweep(nb, npl, 8, d) - np.array([8 * nb, 0])
    elif op == "apply":
        w = _sweep(nb, npl, b, d) - np.array([2 * b * nb, 0])
    else:
        net = 2 * (31 * 64 + 64 * 64 + 64)
        w = np.array([(4 + 4 + 16) * nb, net * nb])
        if op == "mlp_grad":
            w = 3 * w + 2 * _sweep(nb, npl, 4, 3)
    return dict(bytes=float(w[0]), flops=float(w[1]))


# ----------------------------------------------------------------- 64 bits, plain torch
def _closest(kind, params, x):
    """(cp, squared distance) of points x (N, d), FP64."""
    if kind in ("circle", "sphere"):
        r = torch.sqrt((x * x).sum(1))
        return x * (params[0] / r)[:, None], (r - params[0]) ** 2
    if kind == "torus":
        R, rr = params
        rho = torch.sqrt(x[:, 0] ** 2 + x[:, 1] ** 2)
        a = rho - R
        q = torch.sqrt(a * a + x[:, 2] ** 2)
        s = rr / q
        k = (R + a * s) / rho
        return torch.stack([x[:, 0] * k, x[:, 1] * k, x[:, 2] * s], 1), (q - rr) ** 2
    a = torch.tensor(params, dtype=torch.float64, device=x.device)
    ax = x.abs() * a
    lo = torch.full_like(x[:, 0], -float((a * a).min()))
    hi = torch.sqrt((ax * ax).sum(1)) + 1e-300
    for _ in range(90):
        mid = 0.5 * (lo + hi)
        up = ((ax / (a * a + mid[:, None])) ** 2).sum(1) > 1
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    cp = a * a * x / (a * a + (0.5 * (lo + hi))[:, None])
    return cp, ((x - cp) ** 2).sum(1)


def _near(kind, params, x, w):
    """Points that may lie within w of the surface (a superset)."""
    if kind == "ellipsoid":
        a = torch.tensor(params, dtype=torch.float64, device=x.device)
        return min(params) * (torch.sqrt(((x / a) ** 2).sum(1)) - 1).abs() <= w
    return _closest(kind, params, x)[1] <= w * w


def _cubic(s):
    return [-s * (s - 1) * (s - 2) / 6, (s + 1) * (s - 1) * (s - 2) / 2, -(s + 1) * s * (s - 2) / 2,
            (s + 1) * s * (s - 1) / 6]


class _Level:
    """Band, ghost ring and operators of one spacing, in the library's point order:
    4^d bricks in Morton order, nodes of a brick x-fastest, B first, then the ring."""

    def __init__(self, kind, params, inv_dx, form="mbr"):
        self.kind, self.form = kind, form
        self.d = d = 2 if kind == "circle" else 3
        self.h = 1.0 / inv_dx
        self.n = n = 4 * inv_dx + 1
        lam2 = 13.0 if d == 2 else 17.0
        dev = "cuda"
        found = []
        ax = torch.arange(n, device=dev)
        slab = n if d == 2 else max(1, (1 << 24) // (n * n))
        for z0 in range(0, 1 if d == 2 else n, slab):
            zs = ax[z0:z0 + slab] if d == 3 else ax[:1]
            g = torch.stack(torch.meshgrid(zs, ax, ax, indexing="ij"), -1).reshape(-1, 3).flip(1)[:, :d]
            x = -2.0 + g.double() * self.h
            m = _near(kind, params, x, (math.sqrt(lam2) + 1e-6) * self.h)
            g, x = g[m], x[m]
            found.append(g[_closest(kind, params, x)[1] <= lam2 * (self.h * self.h)])
        band = torch.cat(found)
        self.map = torch.full((n ** d,), -1, dtype=torch.int32, device=dev)
        band = band[self._order(band)]
        self.nb = band.shape[0]
        self.map[self._lin(band)] = torch.arange(self.nb, dtype=torch.int32, device=dev)
        ring = torch.cat([self._lin(band) + s for s in self._steps()])
        ring = torch.unique(ring[self.map[ring] < 0])
        g = torch.stack([(ring // n ** a) % n for a in range(d)], 1)
        g = g[self._order(g)]
        self.map[self._lin(g)] = self.nb + torch.arange(g.shape[0], dtype=torch.int32, device=dev)
        self.ijk = torch.cat([band, g])
        self.cp = _closest(kind, params, -2.0 + self.ijk.double() * self.h)[0]
        t = (self.cp + 2.0) / self.h
        self.base = torch.floor(t).long()
        self.s = t - self.base
        self.w = [_cubic(self.s[:, a]) for a in range(d)]
        self.nbr = [self.map[self._lin(self.ijk[: self.nb]) + s].long() for s in self._steps()]
        self.ih2, self.gamma = 1.0 / self.h ** 2, 2.0 * d / self.h ** 2
        if form == "paper":  # band-restricted Laplacian: neighbours outside B dropped
            self.inb = [k < self.nb for k in self.nbr]

    def _steps(self):
        return [s * self.n ** a for a in range(self.d) for s in (-1, 1)]

    def _lin(self, g):
        return sum(g[:, a] * self.n ** a for a in range(self.d))

    def _order(self, g):
        key = torch.zeros_like(g[:, 0])
        for bit in range(9):
            for a in range(self.d):
                key |= ((g[:, a] >> (2 + bit)) & 1) << (2 * self.d + bit * self.d + a)
        for a in range(self.d):
            key |= (g[:, a] & 3) << (2 * a)
        return torch.argsort(key)

    def _cells(self, width, first):
        """Offsets (per axis) of a tensor-product stencil of `width` nodes, z outermost."""
        r = range(width)
        return [(a, b, c) for c in (r if self.d == 3 else [0]) for b in r for a in r]

    def stencil(self, j, width, first):
        """[(band index of a stencil node, its offsets)] of points j of B+."""
        lin = self._lin(self.base[j] + first)
        for o in self._cells(width, first):
            yield self.map[lin + sum(o[a] * self.n ** a for a in range(self.d))].long(), o

    def interp(self, u, j, ref=None):
        """Cubic interpolation of u (or of u - ref) at cp of points j of B+."""
        out = torch.zeros(self.base[j].shape[0], dtype=torch.float64, device=u.device)
        for k, o in self.stencil(j, 4, -1):
            w = self.w[0][o[0]][j]
            for a in range(1, self.d):
                w = w * self.w[a][o[a]][j]
            out = out + w * (u[k] if ref is None else u[k] - ref)
        return out

    def extend(self, u, n):
        parts = [self.interp(u, slice(i, min(i + (1 << 21), n))) for i in range(0, n, 1 << 21)]
        return torch.cat(parts)

    def apply(self, u):
        if self.form == "paper":
            v = -self.gamma * u
            for k, ok in zip(self.nbr, self.inb):
                v = v + self.ih2 * torch.where(ok, u[torch.where(ok, k, 0)], 0.0)
            e1 = torch.zeros_like(u)
            j = slice(0, self.nb)
            for k, o in self.stencil(j, 2, 0):
                w = 1.0
                for a in range(self.d):
                    sa = self.s[j, a]
                    w = w * (sa if o[a] else 1 - sa)
                e1 += w * v[k]
            return e1 - self.gamma * (u - self.extend(u, self.nb))
        w = self.extend(u, self.ijk.shape[0])
        wi = w[: self.nb]
        s = torch.zeros_like(u)
        for k in self.nbr:
            s = s + (w[k] - wi)
        return s * self.ih2 + self.gamma * (wi - u)

    def apply_close(self, u):
        """M u with every difference taken from the point's own value."""
        out = []
        for i in range(0, self.nb, 1 << 20):
            j = torch.arange(i, min(i + (1 << 20), self.nb), device=u.device)
            d0 = self.interp(u, j, u[j])
            s = sum(self.interp(u, k[j], u[j]) - d0 for k in self.nbr)
            out.append(s * self.ih2 + self.gamma * d0)
        return torch.cat(out)

    def diagonal(self):
        """diag(M)."""
        own = self.ijk[: self.nb]
        dm = torch.zeros(self.nb, dtype=torch.float64, device=own.device)
        if self.form == "paper":
            j = slice(0, self.nb)
            for k, o in self.stencil(j, 2, 0):
                w = 1.0
                for a in range(self.d):
                    sa = self.s[j, a]
                    w = w * (sa if o[a] else 1 - sa)
                dist = (self.ijk[k] - own).abs().sum(1)
                dm += w * (torch.where(dist == 0, -self.gamma, 0.0) + torch.where(dist == 1, self.ih2, 0.0))
            return dm - self.gamma * (1 - self._weight_of(own, torch.arange(self.nb, device=own.device)))
        for k in self.nbr:
            dm += self.ih2 * self._weight_of(own, k)
        return dm - self.gamma

    def _weight_of(self, node, k):
        """Weight of a grid node in the cubic stencil of point k of B+."""
        w = torch.ones(node.shape[0], dtype=torch.float64, device=node.device)
        for a in range(self.d):
            off = node[:, a] - self.base[k, a] + 1
            wa = torch.stack([v[k] for v in self.w[a]], 1)
            w = w * torch.where((off >= 0) & (off <= 3), wa.gather(1, off.clamp(0, 3)[:, None])[:, 0], 0.0)
        return w

    def sweeps(self, f, u, count, omega, c=1.0):
        wd = omega / (c - self.diagonal())
        for _ in range(count):
            u = u + wd * (f - c * u + self.apply(u))
        return u


def _linear(src, cp, u):
    """Linear interpolation of the source level's u at points cp."""
    t = (cp + 2.0) / src.h
    b = torch.floor(t).long()
    s = t - b
    lin = src._lin(b)
    out = torch.zeros(cp.shape[0], dtype=torch.float64, device=u.device)
    for o in src._cells(2, 0):
        w = 1.0
        for a in range(src.d):
            w = w * (s[:, a] if o[a] else 1 - s[:, a])
        out += w * u[src.map[lin + sum(o[a] * src.n ** a for a in range(src.d))].long()]
    return out


class _Cycle:
    """The closest-point V-cycle with a direct coarsest solve, c = 1."""

    def __init__(self, kind, params, inv_dx, coarsest, nu, omega, residual):
        self.nu, self.residual = nu, residual
        self.L = []
        while True:
            lv = _Level(kind, params, inv_dx)
            lv.wd = omega / (1.0 - lv.diagonal())
            self.L.append(lv)
            if inv_dx % 2 or inv_dx // 2 < coarsest:
                break
            inv_dx //= 2
        lv = self.L[-1]
        n = lv.nb
        dense = torch.float64 if n <= 10000 else torch.float32
        A = torch.zeros(n, n, dtype=dense, device="cuda")
        row = torch.arange(n, device="cuda")
        A[row, row] = 1.0 + lv.gamma
        for k in lv.nbr:
            for q, o in lv.stencil(k, 4, -1):
                w = lv.w[0][o[0]][k]
                for a in range(1, lv.d):
                    w = w * lv.w[a][o[a]][k]
                A.index_put_((row, q), (-lv.ih2 * w).to(dense), accumulate=True)
        self.lu = torch.linalg.lu_factor(A)
        self.dense = dense

    def coarse(self, f):
        lv = self.L[-1]
        x = torch.zeros_like(f)
        for _ in range(2 if self.dense == torch.float64 else 8):
            r = f - x + lv.apply(x)
            x = x + torch.linalg.lu_solve(*self.lu, r.to(self.dense)[:, None])[:, 0].double()
        return x

    def __call__(self, f, u, l=0):
        if l == len(self.L) - 1:
            return self.coarse(f)
        lv, cv = self.L[l], self.L[l + 1]
        for _ in range(self.nu):
            u = u + lv.wd * (f - u + lv.apply(u))
        e = lv.extend(u, lv.nb) if self.residual == "extended" else u
        r = f - e + lv.apply(e)
        cf = _linear(lv, cv.cp[: cv.nb], r)
        cu = self(cf, torch.zeros_like(cf), l + 1)
        u = u + _linear(cv, lv.cp[: lv.nb], cu)
        for _ in range(self.nu):
            u = u + lv.wd * (f - u + lv.apply(u))
        return u

    def solve(self, f):
        u = torch.zeros_like(f)
        r, last = f, math.inf
        for _ in range(40):
            u = u + self(r, torch.zeros_like(f))
            r = f - u + self.L[0].apply(u)
            now = float(r.abs().max() / f.abs().max())
            if now < 2e-13 or now > 0.7 * last:
                break
            last = now
        return u


def _net(lv, theta, r):
    """The network's correction on residual r: features over the 3^3 neighbourhood."""
    nb = lv.nb
    own = lv.ijk[:nb]
    cols = []
    for c in (-1, 0, 1):
        for b in (-1, 0, 1):
            for a in (-1, 0, 1):
                g = own + torch.tensor([a, b, c], device=own.device)
                k = lv.map[lv._lin(g)].long()
                cols.append(torch.where((k >= 0) & (k < nb), r[k.clamp(0, nb - 1)], 0.0))
    x = torch.stack(cols, 1)
    s = x.abs().amax(1)
    x = x * torch.where(s > 0, 1 / s, 0.0)[:, None]
    off = (-2.0 + own.double() * lv.h - lv.cp[:nb]) / lv.h
    x = torch.cat([x, off, (lv.h ** 2 * lv.diagonal())[:, None], torch.zeros_like(s)[:, None]], 1)
    w1, b1, w2, b2, w3, b3 = torch.split(theta, [2048, 64, 4096, 64, 64, 1])
    h = torch.relu(x @ w1.reshape(32, 64) + b1)
    h = torch.relu(h @ w2.reshape(64, 64) + b2)
    return s * lv.h ** 2 * (h @ w3 + b3)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        out = []
        for i, (axes, inv_dx) in enumerate(_ellipsoids(case)):
            reach = min(axes) ** 2 / max(axes)
            coarsest = inv_dx
            while coarsest % 2 == 0 and (math.sqrt(17.0) + 1) * 2 / coarsest < reach:
                coarsest //= 2
            V = _Cycle("ellipsoid", axes, inv_dx, coarsest, 3, 0.8, "plain")
            y = V.L[0].cp[: V.L[0].nb]
            out += [V.solve(_rhs(y, 1000 * seed + 100 * i + 10 * k)) for k in range(case["n_rhs"])]
            del V
        return out
    kind, params, inv_dx = case["surface"], _params(case), case["inv_dx"]
    if op in ("solve", "cold"):
        V = _Cycle(kind, params, inv_dx, case["coarsest"], 3, 0.8, "plain")
        return V.solve(_rhs(V.L[0].cp[: V.L[0].nb], seed))
    if op == "vcycle":
        V = _Cycle(kind, params, inv_dx, case["coarsest"], case["nu"], case["omega"], case["residual"])
        f = _residual_like(V.L[0].cp[: V.L[0].nb], seed).to(FP[case["prec"]]).double()
        return V(f, torch.zeros_like(f))
    lv = _Level(kind, params, inv_dx, case.get("form", "mbr"))
    y = lv.cp[: lv.nb]
    if op in ("mlp", "mlp_grad"):
        theta = torch.from_numpy(_network(seed)).cuda().double()
        r = _residual_like(y, seed).float().double()
        if op == "mlp":
            return _net(lv, theta, r)
        theta.requires_grad_()
        du = _net(lv, theta, r)
        z = r - (_variable_c(y) * du - lv.apply(du))
        loss = (z * z).sum() / (r * r).sum()
        loss.backward()
        return [float(loss), theta.grad]
    dt = FP[case.get("prec", "f64")]
    if op == "apply":
        return lv.apply(_iterate(y, seed).to(dt).double())
    if op == "residual":
        u = _iterate(y, seed)
        return _rhs(y, seed) - u + lv.apply_close(u)
    f = _residual_like(y, seed).to(dt).double()
    u = (1e-3 * _iterate(y, seed)).to(dt).double()
    return lv.sweeps(f, u, case["sweeps"], case["omega"])
