"""Cases that stand for the work of this framework: Born solves of the acoustic Helmholtz equation through its
public entry points, over the grids, precisions and directions that its users run.

A case is a dict of plain values.  "kind" says which call it is:

    solve     solve_forward to a residual tolerance on a kept solver (float32 iterations, float64 refinement)
    iterate   solve_forward / solve_adjoint of a fixed number of float32 iterations on a kept solver: a slice of a
              long solve on a grid whose whole solve takes seconds to minutes
    solve64   solve_forward to a residual tolerance, all in float64
    apply     (L+I)^-1 or A_s of one field on a kept float64 solver: the step-level calls of a user's own iteration
    gradient  fields of several sources and the medium gradient of a receiver misfit through torch.autograd
    serve     a burst of requests through the continuous-batching server, each with its own medium

Grid extents n0 (fastest), n1, n2 (0 in 2D) are among the supported ones.  Fields of a float32 solve are kept in
single precision by the program that goes on with them, so they are returned as complex64; float64 calls return
complex128.
"""
from __future__ import annotations

import math

import torch

from paper_2507_16087_gb300 import cbs
from paper_2507_16087_gb300 import serving
from paper_2507_16087_gb300 import workloads as W
from paper_2507_16087_gb300.autograd import helmholtz_fields, receiver_misfit

SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 1024, 2048)
LARGEST = 512 ** 3 * 24  # voxel-iterations of the largest case


def _case(kind, n0, n1, n2=0, **kw):
    return dict(kind=kind, n0=n0, n1=n1, n2=n2, **kw)


def listed():
    return [
        # one (L+I)^-1 apply on a small float64 grid: latency and launches
        dict(_case("apply", 32, 24, 16, op="green", adjoint=False), name="green-32x24x16-f64"),
        # the scaled operator of a float64 residual on an ordinary grid, ragged extents
        dict(_case("apply", 128, 96, 192, op="operator", adjoint=False), name="operator-128x96x192-f64"),
        # 2D disc of the examples: a small solve, bound by launches
        dict(_case("solve", 128, 128, medium="inclusion", ppw=6.0, nabs=16), name="solve-128sq"),
        # a 2D request of the serving mix
        dict(_case("solve", 1024, 1024, medium="random", ppw=6.0, nabs=16), name="solve-1024sq"),
        # the small 3D request of the serving mix
        dict(_case("solve", 64, 64, 64, medium="random", ppw=6.0, nabs=10), name="solve-64cube"),
        # the benchmark's own grid: a sphere in water, solved to 1e-6
        dict(_case("solve", 128, 128, 128, medium="inclusion", ppw=6.0, nabs=20), name="solve-128cube"),
        # an odd-shaped 3D grid with factors of three, as a region of interest has it; the adjoint direction
        dict(_case("iterate", 192, 96, 256, adjoint=True, iters=100, ppw=6.0, nabs=16), name="adjoint-192x96x256"),
        # the largest 2D grid of the serving mix
        dict(_case("iterate", 2048, 2048, adjoint=False, iters=100, ppw=6.0, nabs=16), name="iterate-2048sq"),
        # transcranial scale: a slice of the 512^3 solve
        dict(_case("iterate", 512, 512, 512, adjoint=False, iters=24, ppw=6.0, nabs=24), name="iterate-512cube"),
        # all in float64, for those who want no float32 iterations
        dict(_case("solve64", 64, 48, 96, ppw=6.0, nabs=8), name="solve64-64x48x96"),
        # an inversion step: two sources, 64 receivers, gradient in sound speed and density
        dict(_case("gradient", 64, 64, 64, sources=2, ppw=6.0, nabs=10), name="gradient-64cube"),
        # a burst of four requests of different grids
        dict(kind="serve", shapes="64x64x64,512x512,96x96x96,64x64x64", name="serve-4"),
    ]


def _voxels(c):
    return c["n0"] * c["n1"] * max(1, c["n2"])


def _extents(rng, dim, lo, hi, sizes):
    """dim extents of `sizes` whose product lies in [lo, hi], the product spread over its logarithm."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    for _ in range(1000):
        n = [rng.choice(sizes) for _ in range(dim)]
        if target / 1.6 <= math.prod(n) <= target * 1.6 and lo <= math.prod(n) <= hi:
            return n + [0] * (3 - dim)
    return [64] * dim + [0] * (3 - dim)


def draw(rng):
    kind = rng.choice(("solve", "solve", "iterate", "iterate", "solve64", "apply", "gradient"))
    dim = rng.choice((2, 3, 3))
    ppw = round(rng.uniform(4.0, 8.0), 2)
    if kind == "solve":
        if dim == 2:
            n = _extents(rng, 2, 96 * 96, 1 << 20, [s for s in SIZES if s >= 64])
        else:
            n = _extents(rng, 3, 48 ** 3, 1 << 21, [s for s in SIZES if 32 <= s <= 256])
        return _case(kind, *n, medium=rng.choice(("inclusion", "random")), ppw=ppw, nabs=rng.choice((8, 10, 12)))
    if kind == "iterate":
        if dim == 2:
            n = _extents(rng, 2, 1 << 12, 1 << 22, [s for s in SIZES if s >= 32])
        else:
            n = _extents(rng, 3, 1 << 15, 1 << 26, [s for s in SIZES if 24 <= s <= 512])
        iters = min(int(round(math.exp(rng.uniform(math.log(20), math.log(150))))), LARGEST // math.prod(n[:dim]))
        return _case(kind, *n, adjoint=rng.random() < 0.5, iters=iters, ppw=ppw, nabs=rng.choice((4, 6, 8)))
    if kind == "solve64":
        if dim == 2:
            n = _extents(rng, 2, 64 * 64, 1 << 16, [s for s in SIZES if 48 <= s <= 512])
        else:
            n = _extents(rng, 3, 32 ** 3, 1 << 17, [s for s in SIZES if 24 <= s <= 128])
        return _case(kind, *n, ppw=ppw, nabs=rng.choice((6, 8)))
    if kind == "apply":
        if dim == 2:
            n = _extents(rng, 2, 64, 1 << 22, SIZES)
        else:
            n = _extents(rng, 3, 512, 1 << 23, [s for s in SIZES if s <= 512])
        return _case(kind, *n, op=rng.choice(("green", "operator")), adjoint=rng.random() < 0.5)
    n = _extents(rng, 3, 32 ** 3, 1 << 18, [s for s in SIZES if 32 <= s <= 96])
    return _case(kind, *n, sources=rng.choice((1, 2)), ppw=ppw, nabs=rng.choice((8, 10)))


# ------------------------------------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _shape(c):
    return (c["n1"], c["n0"]) if not c["n2"] else (c["n2"], c["n1"], c["n0"])


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, n=1):
    return (lo + (hi - lo) * torch.rand(n, generator=g, device=g.device, dtype=torch.float64)).tolist()


def _nabs(c, shape):
    """The layer's width on every axis (x first): what the case says, and at most a quarter of the extent."""
    return [min(c["nabs"], n // 4) for n in shape[::-1]]


def _medium(c, seed):
    """c0, rho, alpha (float64, on the GPU), dx, omega, layer widths and gamma_max of a case."""
    shape = _shape(c)
    nabs = _nabs(c, shape)
    dx = W.grid_step(c["ppw"])
    if c.get("medium") == "inclusion":  # water with one ball of tissue or bone, off the centre
        g = _gen(seed)
        cc, rr, aa, off = _uniform(g, 2000.0, 2400.0), _uniform(g, 1400.0, 1800.0), _uniform(g, 1.0, 3.0), None
        off = _uniform(g, -0.05, 0.05, len(shape))
        r2 = torch.zeros(shape, dtype=torch.float64, device=_dev())
        for ax, n in enumerate(shape):
            i = torch.arange(n, dtype=torch.float64, device=_dev()) - n * (0.5 + off[ax])
            r2 = r2 + (i * i).reshape([n if a == ax else 1 for a in range(len(shape))])
        inside = r2 < (0.18 * min(shape)) ** 2
        fill = lambda a, b: torch.where(inside, a, b).to(torch.float64)  # noqa: E731
        c0, rho = fill(cc[0], W.C_WATER), fill(rr[0], W.RHO_WATER)
        alpha = fill(W.db_cm_mhz_to_np_m(aa[0]), 0.0)
    else:  # smoothed random tissue between fat and bone
        p = W.smooth_random_medium_torch(shape, seed=seed, ppw=c["ppw"], n_abs=c["nabs"], device=_dev())
        c0, rho, alpha = p.c0, p.rho, p.alpha
    gmax = W.layer_gamma_max(max(1, min(nabs)), dx) if min(nabs) > 0 else 0.0
    return dict(c0=c0.contiguous(), rho=rho.contiguous(), alpha=alpha.contiguous(), dx=dx, omega=2 * math.pi * W.F0,
                nabs=[[n, n] for n in nabs], gamma_max=gmax)


def _point_source(shape, nabs, seed):
    """A unit pressure source at one interior voxel and a weak force on every velocity component beside it."""
    g = _gen(seed + 7919)
    src = torch.zeros((len(shape) + 1,) + tuple(shape), dtype=torch.complex128, device=_dev())
    at = tuple(int(_uniform(g, a + 1, n - a - 2)[0]) for n, a in zip(shape, nabs[::-1]))
    src[(len(shape),) + at] = 1.0
    ph = _uniform(g, 0.0, 2 * math.pi)[0]
    src[(0,) + at] = 1e-7 * complex(math.cos(ph), math.sin(ph))
    return src


def _random_field(shape, seed):
    g = _gen(seed + 104729)
    return torch.randn((len(shape) + 1,) + tuple(shape), generator=g, dtype=torch.complex128, device=_dev())


def _solver(m, **kw):
    return cbs.solver_create(m["c0"], m["rho"], m["alpha"], m["dx"], m["omega"], m["nabs"], m["gamma_max"], **kw)


_TOL = {"solve": 1e-6, "solve64": 1e-8, "gradient": 1e-8, "serve": 1e-6}


def _receivers(shape, nabs):
    """An 8 x 8 (or 8 x 1) set of receivers on the plane two cells inside the layer of the last axis."""
    ix = torch.linspace(nabs[0] + 2, shape[-1] - nabs[0] - 3, 8).round().long()
    iy = torch.linspace(nabs[1] + 2, shape[-2] - nabs[1] - 3, 8).round().long()
    YY, XX = torch.meshgrid(iy, ix, indexing="ij")
    z = torch.full((64,), nabs[2] + 2, dtype=torch.long)
    return tuple(t.reshape(-1).to(_dev()) for t in (z, YY, XX))


def _observed(shape, sources, rec, m):
    """Data of the receivers: the spherical wave of each source in water, a tenth stronger than what it sends."""
    k = m["omega"] / W.C_WATER
    D = len(shape)
    out = []
    for s in sources:
        at = torch.nonzero(s[D])[0]
        r = m["dx"] * torch.sqrt(sum((t - a).double() ** 2 for t, a in zip(rec, at)) + 1.0)
        out.append(1.1 * (m["omega"] / W.C_WATER ** 2) * m["dx"] ** 3 * torch.exp(-1j * k * r) / (4 * math.pi * r))
    return torch.stack(out)


def _serve_requests(c, seed):
    """Requests as serving.make_requests gives them, of the case's grids, all queued at once."""
    reqs = []
    for i, text in enumerate(c["shapes"].split(",")):
        shape = tuple(int(v) for v in text.split("x"))
        g = _gen(seed * 31 + i)
        pos = tuple(int(_uniform(g, 18, n - 18)[0]) for n in shape[::-1])
        r = serving.Request(rid=i, arrival=0.0, shape=shape, ppw=5.0 + i, seed=seed * 31 + i, src_pos=pos)
        r.problem = serving.build_problem(r, 16, _dev())
        reqs.append(r)
    return reqs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        reqs = _serve_requests(case, seed)
        torch.cuda.synchronize()  # the media are there before the requests arrive
        return dict(case=case, server=serving.Server(tol=_TOL["serve"], keep_results=True), requests=reqs)
    shape = _shape(case)
    st = dict(case=case)
    if kind == "apply":
        m = _medium(dict(case, ppw=6.0, nabs=min(8, min(shape) // 4)), seed)
        st["solver"] = _solver(m, precision="fp64")
        st["x"] = _random_field(shape, seed)
        st["out"] = torch.empty_like(st["x"])
        return st
    m = _medium(case, seed)
    nabs = _nabs(case, shape)
    if kind == "gradient":
        src = torch.stack([_point_source(shape, nabs, seed + 1000 * k) for k in range(case["sources"])])
        rec = _receivers(shape, nabs)
        st.update(m=m, sources=src, rec=rec, data=_observed(shape, src, rec, m))
        return st
    st["src"] = _point_source(shape, nabs, seed)
    st["field"] = torch.empty_like(st["src"])
    if kind == "solve":
        st["solver"] = _solver(m, precision="fp32_refine", tol=_TOL[kind])
    elif kind == "iterate":
        st["solver"] = _solver(m, precision="fp32", tol=0.0, max_iter=case["iters"])
    else:
        st["solver"] = _solver(m, precision="fp64", tol=_TOL[kind])
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        state["server"].run(state["requests"], realtime=False)
        return [r.result.to(torch.complex64) for r in state["requests"]]
    if kind == "apply":
        s = state["solver"]
        (s.green_apply if case["op"] == "green" else s.operator_apply)(state["x"], state["out"], case["adjoint"])
        return state["out"]
    if kind == "gradient":
        m = state["m"]
        c0, rho = m["c0"].clone().requires_grad_(), m["rho"].clone().requires_grad_()
        f = helmholtz_fields(c0, rho, m["alpha"], state["sources"], m["dx"], m["omega"], m["nabs"], m["gamma_max"],
                             tol=_TOL[kind])
        J = receiver_misfit(f, state["data"], state["rec"])
        J.backward()
        # the update of the medium is made in single precision
        return {"misfit": J.detach().float(), "grad_c0": c0.grad.float(), "grad_rho": rho.grad.float(),
                "fields": f.detach().to(torch.complex64)}
    s = state["solver"]
    solve = s.solve_adjoint if case.get("adjoint") else s.solve_forward
    solve(state["src"], state["field"])
    return state["field"] if kind == "solve64" else state["field"].to(torch.complex64)


# ------------------------------------------------------------------------------------------------ what a pass needs
# Born iterations to the tolerance for media of these ranges, to the nearest few hundred (the count depends on the
# contrast and the grid, and a case's work is stated for this many)
_ITERS = {"solve": 1000, "solve64": 1000, "gradient": 1500, "serve": 1000}


def _fft_flops(n, C):
    """Forward and inverse transforms of C components along every axis: 5 N log2 N each."""
    return 2 * C * 5 * math.prod(n) * sum(math.log2(v) for v in n)


def work(case):
    """One iteration reads x, y and the medium and writes x; its transforms, the symbol (about 100 flops a voxel) and
    the update.  An apply reads and writes one field."""
    kind = case["kind"]
    if kind == "serve":
        w = [work(_case("solve", *(int(v) for v in reversed(t.split("x"))))) for t in case["shapes"].split(",")]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    n = [case[k] for k in ("n0", "n1", "n2") if case[k]]
    N, D, C = math.prod(n), len(n), len(n) + 1
    flops = _fft_flops(n, C) + 100 * N
    if kind == "apply":
        return {"bytes": 2 * C * N * 16, "flops": flops}
    size = 16 if kind == "solve64" else 8
    per = N * (3 * C * size + (D + 2) * size // 2)
    passes = case["iters"] if kind == "iterate" else _ITERS[kind] * (2 * case["sources"] if kind == "gradient" else 1)
    return {"bytes": passes * per, "flops": passes * flops}


# ------------------------------------------------------------------------------------------------ 64-bit values
class _Plain:
    """The scaled system of the method in plain torch, 64 bits: A_s = L + V, one Born step, and the solve."""

    def __init__(self, m, shape, nu=0.8, beta=0.95):
        self.shape, self.D, self.nu, self.m = shape, len(shape), nu, m
        D, om = self.D, m["omega"]
        gc, gs, self.t, self.k2 = [], [], [], 0
        for a, n in enumerate(shape[::-1]):  # axis a of the grid (x first) is tensor axis D - 1 - a
            i = torch.arange(n, dtype=torch.float64, device=_dev())
            lo, hi = m["nabs"][a]

            def layer(xi):
                d = torch.zeros_like(xi)
                if lo:
                    d = torch.maximum(d, (lo - xi) / lo)
                if hi:
                    d = torch.maximum(d, (xi - (n - 1 - hi)) / hi)
                return m["gamma_max"] * d.clamp(max=1.0) ** 2

            view = [n if ax == D - 1 - a else 1 for ax in range(D)]
            gc.append(layer(i).reshape(view))
            gs.append(layer(i + 0.5).reshape(view))
            k = 2 * math.pi * torch.fft.fftfreq(n, m["dx"], dtype=torch.float64, device=_dev())
            self.t.append((k * torch.exp(0.5j * k * m["dx"])).reshape(view))
            self.k2 = self.k2 + (k * k).reshape(view)
        self.gc = sum(gc[1:], gc[0]).expand(shape)
        self.gs = [sum((gs[b] if b == e else gc[b] for b in range(1, D)), gs[0] if e == 0 else gc[0]).expand(shape)
                   for e in range(D)]
        d, q, _ = self.diagonal(m["c0"], m["rho"])
        mid = lambda zs: 0.5 * complex(min(float(z.real.min()) for z in zs) + max(float(z.real.max()) for z in zs),  # noqa: E731
                                       min(float(z.imag.min()) for z in zs) + max(float(z.imag.max()) for z in zs))
        self.a1, self.a2 = mid(d), mid([q])
        self.l1 = max(float((z - self.a1).abs().max()) for z in d) / beta
        self.l2 = float((q - self.a2).abs().max()) / beta
        self.B = [1 - (z - self.a1) / self.l1 for z in d] + [1 - (q - self.a2) / self.l2]
        self.om = om

    def diagonal(self, c0, rho):
        """The system's diagonal: staggered density times (i omega + gamma), (i omega + gamma) / (rho c^2), and 1 / (rho c^2)."""
        m, om = self.m, self.m["omega"]
        ic2 = (1 - 2j * m["alpha"] * c0 / om) / (rho * c0 * c0)
        d = []
        for e in range(self.D):
            rs = 0.5 * (rho + torch.roll(rho, -1, dims=self.D - 1 - e))
            d.append(rs * torch.complex(self.gs[e], torch.full_like(self.gs[e], om)))
        return d, ic2 * torch.complex(self.gc, torch.full_like(self.gc, om)), ic2

    def source(self, s, adjoint=False):
        """The scaled right-hand side of a physical source."""
        f = [self.l1 ** -0.5] * self.D + [self.l2 ** -0.5]
        if adjoint:
            return torch.stack([s[c] * f[c] for c in range(self.D + 1)])
        rho = self.m["rho"]
        ic2 = self.diagonal(self.m["c0"], rho)[2]
        y = [0.5 * (rho + torch.roll(rho, -1, dims=self.D - 1 - e)) * s[e] * f[e] for e in range(self.D)]
        return torch.stack(y + [ic2 * s[self.D] * f[self.D]])

    def field(self, x):
        f = [self.l1 ** -0.5] * self.D + [self.l2 ** -0.5]
        for c in range(self.D + 1):
            x[c] *= f[c]
        return x

    def green(self, v, adjoint=False):
        """(L + I)^-1 v by elimination of the velocity, wavenumber by wavenumber (v is overwritten)."""
        dims = tuple(range(1, self.D + 1))
        w = torch.fft.fftn(v, dim=dims)
        al, be, g = self.a1 / self.l1 + 1, self.a2 / self.l2 + 1, 1j / math.sqrt(self.l1 * self.l2)
        if adjoint:
            al, be, g = al.conjugate(), be.conjugate(), g.conjugate()
        rhs = w[self.D].clone()
        for e in range(self.D):
            rhs -= g / al * self.t[e].conj() * w[e]
        p = rhs / (be - g * g / al * self.k2)
        for e in range(self.D):
            w[e] = (w[e] - g * self.t[e] * p) / al
        w[self.D] = p
        del rhs, p
        return torch.fft.ifftn(w, dim=dims)

    def operator(self, x, adjoint=False):
        dims = tuple(range(1, self.D + 1))
        g = 1j / math.sqrt(self.l1 * self.l2) * (-1 if adjoint else 1)
        w = torch.fft.fftn(x, dim=dims)
        out = torch.empty_like(w)
        out[self.D] = sum(g * self.t[e].conj() * w[e] for e in range(self.D))
        for e in range(self.D):
            out[e] = g * self.t[e] * w[self.D]
        out = torch.fft.ifftn(out, dim=dims)
        for c in range(self.D + 1):  # a / lambda + V = the diagonal over lambda
            b = 1 - self.B[c] + (self.a1 / self.l1 if c < self.D else self.a2 / self.l2)
            out[c] += (b.conj() if adjoint else b) * x[c]
        return out

    def step(self, x, y, adjoint=False):
        b = [z.conj() if adjoint else z for z in self.B]
        z = self.green(torch.stack([b[c] * x[c] + y[c] for c in range(self.D + 1)]), adjoint)
        for c in range(self.D + 1):
            z[c] -= x[c]
            z[c] *= b[c] * self.nu
        x += z
        return x

    def solve(self, y, tol=1e-10, adjoint=False, most=20000):
        x = torch.zeros_like(y)
        ny = float(torch.linalg.vector_norm(y))
        for it in range(1, most + 1):
            x = self.step(x, y, adjoint)
            if it % 100 == 0 and float(torch.linalg.vector_norm(y - self.operator(x, adjoint))) <= tol * ny:
                break
        return x


def _exact_gradient(case, seed):
    st = prepare(case, seed)
    m, shape = st["m"], _shape(case)
    P = _Plain(m, shape)
    D = P.D
    X = torch.stack([P.field(P.solve(P.source(s))) for s in st["sources"]])
    at = (slice(None), D) + tuple(st["rec"])
    miss = X[at] - st["data"]
    c0, rho = m["c0"].clone().requires_grad_(), m["rho"].clone().requires_grad_()
    total = 0.0
    for k, s in enumerate(st["sources"]):
        g = torch.zeros_like(X[k])
        g[at[1:]] = miss[k]
        lam = P.field(P.solve(P.source(g, True), adjoint=True))
        # Re <lambda, b(m) - A(m) X>: only the diagonal and the right-hand side depend on the medium
        d, q, ic2 = P.diagonal(c0, rho)
        for e in range(D):
            rs = 0.5 * (rho + torch.roll(rho, -1, dims=D - 1 - e))
            total = total + (lam[e].conj() * (rs * s[e] - d[e] * X[k, e])).real.sum()
        total = total + (lam[D].conj() * (ic2 * s[D] - q * X[k, D])).real.sum()
    gc, gr = torch.autograd.grad(total, (c0, rho))
    return {"misfit": 0.5 * (miss.abs() ** 2).sum(), "grad_c0": gc, "grad_rho": gr, "fields": X}


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for r in _serve_requests(case, seed):
            p = r.problem
            m = dict(c0=p.c0, rho=p.rho, alpha=p.alpha, dx=p.dx, omega=p.omega, nabs=p.nabs, gamma_max=p.gamma_max)
            P = _Plain(m, r.shape)
            s = torch.zeros((P.D + 1,) + r.shape, dtype=torch.complex128, device=_dev())
            s[(P.D,) + r.src_pos[::-1]] = 1.0
            out.append(P.field(P.solve(P.source(s), tol=1e-8))[P.D])
        return out
    if kind == "gradient":
        return _exact_gradient(case, seed)
    shape = _shape(case)
    if kind == "apply":
        m = _medium(dict(case, ppw=6.0, nabs=min(8, min(shape) // 4)), seed)
        P = _Plain(m, shape)
        x = _random_field(shape, seed)
        return (P.green if case["op"] == "green" else P.operator)(x, case["adjoint"])
    P = _Plain(_medium(case, seed), shape)
    src = _point_source(shape, _nabs(case, shape), seed)
    adjoint = bool(case.get("adjoint"))
    y = P.source(src, adjoint)
    del src
    if kind == "iterate":
        x = torch.zeros_like(y)
        for _ in range(case["iters"]):
            x = P.step(x, y, adjoint)
        return P.field(x)
    return P.field(P.solve(y, tol=1e-9 if kind == "solve" else 1e-12))
