"""What is timed of this framework: FWIME operators as a user's program calls them.

Each case is one operator call (or the pair an inversion makes) through ``paper_2206_02362_gb300.Context``
with the defaults a program would use, on a grid, an acquisition and a record length of the repository's
workloads.  Records of the survey-sized cases are shortened (the cost is linear in nt) and keep their grids,
shots per launch, offsets and receivers.  Inputs are drawn on the GPU from the seed alone: folded layered
velocities, a Ricker source per shot, data made of hyperbolic events plus noise, and p~ made of dipping
reflectors focused around zero offset.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2206_02362_gb300 as fw

DEV = "cuda" if torch.cuda.is_available() else "cpu"
A8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)   # 8th-order second derivative


def _case(name, op, nz, nx, sponge, nt, nh, nshot, dx, dt, f0, lag=0, fs=0, niter=0, graph=0, rec_step=2):
    c = dict(op=op, nz=nz, nx=nx, sponge=sponge, nt=nt, nh=nh, nshot=nshot, dx=dx, dt=dt, f0=f0, lag=lag, fs=fs,
             niter=niter, graph=graph, rec_step=rec_step)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one shot on the tiny grid, a thousand steps of a few microseconds each
        _case("forward_small", "forward", 100, 200, 30, 1000, 1, 1, 10.0, 1e-3, 15.0, rec_step=1),
        # T on a ragged toy problem of the test suite's size (linearised modelling while developing)
        _case("tomo_small", "tomo", 37, 300, 10, 250, 5, 3, 10.0, 1e-3, 20.0, rec_step=3),
        # one forward-modelling request of the serving mix (one shot, odd sizes)
        _case("forward_request", "forward", 401, 1203, 50, 1500, 1, 1, 10.0, 1e-3, 10.0),
        # one gradient request of the serving mix
        _case("gradient_request", "gradient", 300, 900, 50, 1000, 11, 1, 10.0, 1e-3, 10.0),
        # the line search's extra objective evaluation, with a free surface, on a medium problem
        _case("objective_line_search", "objective", 302, 1001, 50, 400, 11, 16, 10.0, 1e-3, 10.0, fs=1),
        # f(m) over all 100 shots of the Marmousi2-shaped survey (the residual of every outer iteration)
        _case("forward_survey", "forward", 350, 1700, 50, 400, 1, 100, 10.0, 8e-4, 8.0),
        # conventional FWI gradient B* r over a North-Sea-shaped survey
        _case("born_adj_survey", "born_adj", 400, 1600, 50, 400, 1, 60, 12.5, 1e-3, 8.0),
        # extended modelling and migration B~, B~* of one VP iteration: the benchmark's step
        _case("pair_survey", "pair", 350, 1700, 50, 400, 21, 100, 10.0, 8e-4, 8.0),
        # the same pair with the time-lag extension
        _case("pair_time_lag", "pair", 350, 1700, 50, 400, 21, 24, 10.0, 8e-4, 8.0, lag=2),
        # FWIME gradient over half the North-Sea-shaped survey, captured in a graph as the benchmark does
        _case("gradient_survey", "gradient", 400, 1600, 50, 300, 31, 60, 12.5, 1e-3, 8.0, graph=1),
        # FWIME gradient of a few shots on the Salt-shaped grid, the largest one
        _case("gradient_salt", "gradient", 1200, 5000, 50, 200, 41, 4, 6.25, 5e-4, 10.0),
        # VP iterations with the 101 offsets at 30 m spacing of the paper's Marmousi2 example
        _case("vp_wide_offsets", "vp", 117, 567, 50, 250, 101, 16, 30.0, 2.5e-3, 8.0, niter=1),
    ]


def draw(rng):
    """One more case: any operator, any size between the listed ones, odd offset counts and ragged grids."""
    def lg(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    while True:
        op = rng.choice(["forward", "forward", "born_adj", "pair", "pair", "gradient", "gradient", "objective", "vp",
                         "tomo"])
        ext = op not in ("forward", "born_adj")
        nz, nx = lg(30, 1200), lg(120, 5000)
        sponge = rng.choice([10, 20, 30, 50, 50, 50])
        nt = lg(120, 2000)
        nshot = lg(1, 100)
        nh = rng.choice([1, 5, 7, 11, 21, 21, 31, 31, 41, 51, 101]) if ext else 1
        lag = rng.choice([0, 0, 0, 1, 2]) if op == "pair" and nh in (5, 11, 21, 31) else 0
        fs = rng.choice([0, 0, 1]) if op in ("forward", "objective") else 0
        dx = rng.choice([6.25, 10.0, 12.5, 25.0, 30.0])
        dt = round(0.55 * 2.0 * dx / (4700.0 * math.sqrt(2 * 6.502)), 5)
        c = _case("", op, nz, nx, sponge, nt, nh, nshot, dx, dt, rng.choice([6.0, 8.0, 10.0]), lag=lag, fs=fs,
                  niter=1 if op == "vp" else 0, rec_step=rng.choice([1, 2, 3]))
        # no more than the largest listed ones: propagations, offset products (dearer where the kernels are
        # generic), device memory (three states at a time) and time steps of launch-bound problems
        pts, phys = _padded(c) * nshot * (nt - 1), float(nz) * nx * nshot * (nt - 1)
        prods = phys * nh * (20 if nh in (7, 51, 101) else 1) * _passes(c)[1]
        fields = 4 + (9 * math.sqrt(nt) + 9 if op != "forward" else 0) + (40 * nh * lag if lag else 0)
        if pts * _passes(c)[0] < 4e10 and 2e8 < pts and prods < 8e11 and _padded(c) * 4 * nshot * fields < 2.4e10 \
                and nh * nz * nx < 2.5e8:
            return c


# ------------------------------------------------------------------ inputs

def _padded(c):
    return (c["nz"] + 2 * (c["sponge"] + 4)) * (c["nx"] + 2 * (c["sponge"] + 4))


def _geometry(c):
    src_ix = np.round(np.linspace(0.03, 0.97, c["nshot"] + 2)[1:-1] * (c["nx"] - 1)).astype(np.int32)
    rec_ix = np.arange(0, c["nx"], c["rec_step"], dtype=np.int32)
    return np.full(c["nshot"], 2, np.int32), src_ix, np.full(len(rec_ix), 2, np.int32), rec_ix


def _inputs(c, seed):
    """The float32 tensors of a case, from the seed alone."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (seed + 1))
    u = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    nz, nx, nt, nh, S = c["nz"], c["nx"], c["nt"], c["nh"], c["nshot"]
    src_iz, src_ix, rec_iz, rec_ix = _geometry(c)
    nrec = len(rec_ix)
    z = torch.arange(nz, device=DEV, dtype=torch.float32)[:, None] / nz
    x = torch.arange(nx, device=DEV, dtype=torch.float32)[None, :] / nx
    # velocity: 12 folded layers from 1.5 to about 4.5 km/s
    bases = torch.sort(0.05 + 0.95 * u(11))[0]
    vels = torch.linspace(1500.0, 4500.0, 12, device=DEV) * (1.0 + 0.04 * (u(12) - 0.5))
    fold = 0.06 * torch.sin(6.2832 * (x * (1.0 + 3.0 * u(1)) + u(1))) * z
    t = {"v": vels[torch.searchsorted(bases, (z + fold).contiguous())].clamp(1450.0, 4600.0).contiguous()}
    # one Ricker wavelet per shot, slightly different amplitudes
    tau = torch.arange(nt, device=DEV, dtype=torch.float32) * c["dt"] - 1.2 / c["f0"]
    a = (math.pi * c["f0"] * tau) ** 2
    t["w"] = ((1.0 - 2.0 * a) * torch.exp(-a) * (0.9 + 0.2 * u(S, 1))).contiguous()
    if c["op"] != "forward" and c["op"] != "tomo":
        # data: hyperbolic events of the source wavelet plus 2 % noise
        off = torch.as_tensor(np.abs(src_ix[:, None].astype(np.float32) - rec_ix[None, :]), device=DEV) * c["dx"]
        d = 1e-3 * torch.randn(S, nt, nrec, generator=g, device=DEV)
        tn = torch.arange(nt, device=DEV, dtype=torch.float32)[None, :, None] * c["dt"]
        T = nt * c["dt"]
        for _ in range(3):
            t0, ve, amp = float(0.15 + 0.6 * u(1)) * T, float(1500.0 + 1500.0 * u(1)), float(0.02 + 0.06 * u(1))
            ar = (math.pi * c["f0"]) ** 2 * (tn - torch.sqrt(t0 ** 2 + (off / ve) ** 2)[:, None, :]) ** 2
            d += amp * (1.0 - 2.0 * ar) * torch.exp(-ar)
        t["d"] = d.contiguous()
    if c["op"] in ("pair", "gradient", "objective", "tomo", "vp"):
        # p~ in m/s: dipping reflectors, decaying away from zero offset, plus noise
        refl = torch.zeros(nz, nx, device=DEV)
        for _ in range(4):
            refl += torch.sin(6.2832 * (z * (4.0 + 20.0 * u(1)) + x * (6.0 * u(1) - 3.0) + u(1)))
        hm = (nh - 1) // 2
        taper = torch.exp(-((torch.arange(nh, device=DEV) - hm) / (0.5 * hm + 0.5)) ** 2)
        t["pt"] = 3.0 * torch.randn(nh, nz, nx, generator=g, device=DEV)
        t["pt"] += 20.0 * refl[None]
        t["pt"] *= taper[:, None, None]
    if c["op"] == "tomo":
        t["dv"] = (40.0 * torch.sin(9.0 * z + 14.0 * x + 6.2832 * u(1)) * torch.sin(3.1416 * z) *
                   torch.sin(3.1416 * x)).contiguous()
    return t


def prepare(case, seed):
    c = case
    t = _inputs(c, seed)
    grid = fw.Grid(nz=c["nz"], nx=c["nx"], sponge=c["sponge"], nt=c["nt"], dt=c["dt"], dx=c["dx"], nh=c["nh"])
    geom = fw.Geometry(*_geometry(c))
    opts = {}
    if c["lag"]:
        opts["time_lag"] = c["lag"]
    if c["fs"]:
        opts["free_surface"] = 1
    if c["op"] == "pair":
        opts["reuse_background"] = 1     # v and w stay the same between B~ and B~*
    stream = None
    if c["graph"]:
        stream = torch.cuda.Stream()
        opts["graph"] = 1
    ctx = fw.Context(grid, geom, stream=stream, **opts)
    shape_d = (c["nshot"], c["nt"], geom.nrec)
    out = {}
    if c["op"] in ("forward", "pair", "tomo"):
        out["data"] = torch.zeros(shape_d, device=DEV)
    if c["op"] == "pair":
        out["image"] = torch.zeros((c["nh"], c["nz"], c["nx"]), device=DEV)
    if c["op"] in ("born_adj", "gradient"):
        out["grad"] = torch.zeros((c["nz"], c["nx"]), device=DEV)
    if c["op"] == "vp":
        out["pt"] = torch.zeros((c["nh"], c["nz"], c["nx"]), device=DEV)
    torch.cuda.synchronize()
    return {"case": c, "ctx": ctx, "stream": stream, "t": t, "out": out}


EPS = 1e-6    # DSO weight of the objective and of the VP problem


def run(state):
    c, ctx, t, out = state["case"], state["ctx"], state["t"], state["out"]
    op = c["op"]
    if op == "forward":
        return ctx.forward(t["v"], t["w"], out["data"])
    if op == "tomo":
        return ctx.tomo(t["v"], t["w"], t["pt"], t["dv"], out["data"])
    if op == "born_adj":
        return ctx.born_adj(t["v"], t["w"], t["d"], out["grad"])
    if op == "pair":
        ctx.born_ext(t["v"], t["w"], t["pt"], out["data"])
        ctx.born_ext_adj(t["v"], t["w"], t["d"], out["image"])
        return out["data"], out["image"]
    if op == "objective":
        return ctx.objective(t["v"], t["w"], t["pt"], t["d"], eps=EPS)
    if op == "gradient":
        J = ctx.gradient(t["v"], t["w"], t["pt"], t["d"], out["grad"], eps=EPS)
        return J, out["grad"]
    out["pt"].zero_()
    hist = ctx.vp_solve(t["v"], t["w"], t["d"], out["pt"], eps=EPS, niter=c["niter"])
    return out["pt"], hist


def _passes(c):
    """(propagations, extension passes) of one run: the propagations of the operators' definitions, the
    source wavefield of an adjoint counted once more (its recomputation from checkpoints)."""
    n = c["niter"]
    return {"forward": (1, 0), "born_adj": (2, 0), "pair": (4, 2), "objective": (2, 1), "gradient": (6, 4),
            "tomo": (4, 3), "vp": (2 + 4 * n, 1 + 2 * n)}[c["op"]]


def work(case):
    """Bytes: 12 per propagated grid point and step (read q^n and q^n-1, write q^n+1) and 8 per physical point
    and step of an extension pass (one field in, one out), plus the inputs and outputs once.  Operations: 35
    per propagated point, 2 nh per extension point."""
    c = case
    props, exts = _passes(c)
    pts = float(_padded(c)) * c["nshot"] * (c["nt"] - 1)
    phys = float(c["nz"]) * c["nx"] * c["nshot"] * (c["nt"] - 1)
    nm, nd = c["nz"] * c["nx"], c["nshot"] * c["nt"] * len(_geometry(c)[3])
    io = 4.0 * (nm * (2 + 2 * c["nh"] * (exts > 0)) + nd)
    return {"bytes": 12.0 * pts * props + 8.0 * phys * exts + io,
            "flops": 35.0 * pts * props + 2.0 * c["nh"] * phys * exts}


# ------------------------------------------------------------------ 64-bit values

class _Wave:
    """The discretisation in float64 with plain tensor operations, `G` shots at a time."""

    def __init__(self, c, v, w):
        f32 = lambda a: float(np.float32(a))  # noqa: E731
        self.c, self.dt, self.dx = c, f32(c["dt"]), f32(c["dx"])
        self.nz, self.nx, self.nt, self.nh = c["nz"], c["nx"], c["nt"], c["nh"]
        W = c["sponge"]
        self.o = o = W + 4
        self.NZ, self.NX = self.nz + 2 * o, self.nx + 2 * o
        self.v, self.w = v.double(), w.double()
        iz = (torch.arange(self.NZ, device=DEV) - o).clamp(0, self.nz - 1)
        ix = (torch.arange(self.NX, device=DEV) - o).clamp(0, self.nx - 1)
        cc = (self.v[iz][:, ix] * self.dt) ** 2

        def taper(N, n):
            i = torch.arange(N, device=DEV, dtype=torch.float64)
            k = torch.clamp(torch.maximum(o - i, i - (o + n - 1)), min=0.0)
            g = torch.exp(-(0.3 * k / max(W, 1)) ** 2)
            g[:4] = 0.0
            g[-4:] = 0.0
            return g
        gz, gx = taper(self.NZ, self.nz), taper(self.NX, self.nx)
        if c["fs"]:       # no sponge above the surface row, which is silent
            gz[:o] = 1.0
            gz[:o - 4] = 0.0
            cc[:o - 4] = 0.0
            cc[o] = 0.0
        self.g = (gz[:, None] * gx[None, :])[4:-4, 4:-4].contiguous()
        self.cc = cc[4:-4, 4:-4].contiguous()
        self.b = 2.0 / self.v ** 3
        siz, six, riz, rix = _geometry(c)
        T = lambda a: torch.as_tensor(np.asarray(a, dtype=np.int64), device=DEV)  # noqa: E731
        self.siz, self.six = T(siz) + o - 4, T(six) + o - 4
        self.rz, self.rx = T(riz) + o, T(rix) + o
        self.rows = slice(o, o + self.nz)

    def field(self, G):
        return torch.zeros(G, self.NZ, self.NX, device=DEV, dtype=torch.float64)

    def lap(self, q, out):
        NZ, NX, s = self.NZ, self.NX, 1.0 / self.dx ** 2
        torch.mul(q[:, 4:-4, 4:-4], 2 * A8[0] * s, out=out)
        for k in range(1, 5):
            a = A8[k] * s
            out.add_(q[:, 4:-4, 4 + k:NX - 4 + k], alpha=a).add_(q[:, 4:-4, 4 - k:NX - 4 - k], alpha=a)
            out.add_(q[:, 4 + k:NZ - 4 + k, 4:-4], alpha=a).add_(q[:, 4 - k:NZ - 4 - k, 4:-4], alpha=a)
        return out

    def march(self, G, source):
        """q^0 .. q^(nt-1); source(n, s) adds s^n to the active region's buffer.  Yields (n, q^n, D^n) for
        n = 0 .. nt-1, D^n (physical rows, all columns) None for the last."""
        q, p = self.field(G), self.field(G)
        lap = torch.empty(G, self.NZ - 8, self.NX - 8, device=DEV, dtype=torch.float64)
        o = self.o
        for n in range(self.nt - 1):
            self.lap(q, lap)
            source(n, lap)
            qi, pi = q[:, 4:-4, 4:-4], p[:, 4:-4, 4:-4]
            D = p[:, self.rows] - 2.0 * q[:, self.rows]
            pi.mul_(-self.g).add_(qi, alpha=2.0).addcmul_(lap, self.cc.expand_as(lap)).mul_(self.g)
            if self.c["fs"]:
                p[:, o] = 0.0
                for k in range(1, 5):
                    p[:, o - k] = -p[:, o + k]
            D.add_(p[:, self.rows]).mul_(1.0 / self.dt ** 2)
            if self.c["fs"]:
                D[:, 0] = 0.0
            yield n, q, D
            q, p = p, q
        yield self.nt - 1, q, None

    def back(self, G, inject):
        """The transposed recursion; inject(n, a) adds to the adjoint of q^n.  Yields (n, source adjoint of
        s^n on the padded grid) for n = nt-2 .. 0."""
        l1, l2 = self.field(G), self.field(G)     # adjoints of q^(n+1), q^(n+2)
        mu = self.field(G)
        lap = torch.empty(G, self.NZ - 8, self.NX - 8, device=DEV, dtype=torch.float64)
        gc, g2 = self.g * self.cc, self.g ** 2
        inject(self.nt - 1, l1)
        for n in range(self.nt - 2, -1, -1):
            torch.mul(l1[:, 4:-4, 4:-4], gc, out=mu[:, 4:-4, 4:-4])
            yield n, mu
            if n == 0:
                return
            self.lap(mu, lap)
            a = l2[:, 4:-4, 4:-4]
            a.mul_(-g2).addcmul_(l1[:, 4:-4, 4:-4], (2.0 * self.g).expand_as(a)).add_(lap)
            # transposed padding: nothing outside the active region
            inject(n, l2)
            l1, l2 = l2, l1

    def point(self, s0, G):
        r, sc = torch.arange(G, device=DEV), 1.0 / self.dx ** 2

        def add(n, s):
            s[r, self.siz[s0:s0 + G], self.six[s0:s0 + G]] += self.w[s0:s0 + G, n] * sc
        return add

    def record(self, q):
        return q[:, self.rz, self.rx]

    def inject(self, d):
        def add(n, a):
            a.view(a.shape[0], -1).index_add_(1, self.rz * self.NX + self.rx, d[:, n])
        return add

    def cols(self, h):
        """Column ranges (physical x, padded x + h) with x + h and x - h inside the padded row."""
        lo = max(0, abs(h) - self.o)
        hi = min(self.nx, self.NX - self.o - abs(h))
        return lo, hi

    def scatter(self, Wt, D, sign=1):
        """Rows of sum_h W(x, h) D(x - sign h) at x + sign h."""
        e, o, hm = torch.zeros_like(D), self.o, (self.nh - 1) // 2
        for i in range(self.nh):
            h = sign * (i - hm)
            lo, hi = self.cols(h)
            if lo < hi:
                e[..., o + lo + h:o + hi + h].addcmul_(D[..., o + lo - h:o + hi - h],
                                                       Wt[i][:, lo:hi].expand_as(D[..., lo:hi]))
        return e

    def image(self, I, D, L):
        """I(x, h) += sum over shots of D(x - h) L(x + h)."""
        o, hm = self.o, (self.nh - 1) // 2
        for i in range(self.nh):
            h = i - hm
            lo, hi = self.cols(h)
            if lo < hi:
                I[i][:, lo:hi].add_((D[..., o + lo - h:o + hi - h] * L[..., o + lo + h:o + hi + h]).sum(0))


def _groups(c, histories):
    per = c["nt"] * c["nz"] * (c["nx"] + 2 * c["sponge"] + 8) * 8.0 * histories + 40 * 8.0 * _padded(c)
    G = int(max(1, min(c["nshot"], 6e10 // per)))
    return [(s, min(G, c["nshot"] - s)) for s in range(0, c["nshot"], G)]


def _forward(W, s0, G, hist=False):
    d, Ds = torch.zeros(G, W.nt, len(W.rx), device=DEV, dtype=torch.float64), []
    for n, q, D in W.march(G, W.point(s0, G)):
        d[:, n] = W.record(q)
        if hist and D is not None:
            Ds.append(D.clone())
    return d, Ds


def _source_rows(W, e):
    """Source callback adding e(n) (physical rows, all columns) to the active region."""
    def add(n, s):
        s[:, W.o - 4:W.o - 4 + W.nz].add_(e(n)[..., 4:-4])
    return add


def _ext_e(W, Wt, Ds):
    hm, L = (W.nh - 1) // 2, W.c["lag"]
    if not L:
        return lambda n: W.scatter(Wt, Ds[n])

    def e(n):
        out = torch.zeros_like(Ds[0])
        for i in range(W.nh):
            m = n - 2 * L * (i - hm)
            if 0 <= m < len(Ds):
                out[..., W.o:W.o + W.nx].addcmul_(Ds[m][..., W.o:W.o + W.nx], Wt[i].expand(out.shape[0], -1, -1))
        return out
    return e


def _born_ext(W, Wt, Ds, G, hist=False):
    d, Dq = torch.zeros(G, W.nt, len(W.rx), device=DEV, dtype=torch.float64), []
    for n, q, D in W.march(G, _source_rows(W, _ext_e(W, Wt, Ds))):
        d[:, n] = W.record(q)
        if hist and D is not None:
            Dq.append(D.clone())
    return d, Dq


def _ext_image(W, I, Ds, d):
    """I += the extended image of the data d (without b)."""
    hm, L = (W.nh - 1) // 2, W.c["lag"]
    for n, mu in W.back(d.shape[0], W.inject(d)):
        if not L:
            W.image(I, Ds[n], mu[:, W.rows])
            continue
        for i in range(W.nh):
            m = n - 2 * L * (i - hm)
            if 0 <= m < len(Ds):
                I[i].add_((Ds[m] * mu[:, W.rows])[..., W.o:W.o + W.nx].sum(0))


def exact(case, seed):
    c = case
    t = _inputs(c, seed)
    W = _Wave(c, t["v"], t["w"])
    op, o, ph = c["op"], W.o, slice(W.o, W.o + W.nx)
    dd = t["d"].double() if "d" in t else None
    pt = t["pt"].double() if "pt" in t else None
    zm = lambda *s: torch.zeros(*s, W.nz, W.nx, device=DEV, dtype=torch.float64)  # noqa: E731
    hm = (W.nh - 1) // 2
    dso = torch.arange(W.nh, device=DEV, dtype=torch.float64).sub_(hm).abs_().add_(1.0)[:, None, None]
    eps = float(np.float32(EPS))
    if op == "forward":
        return torch.cat([_forward(W, s0, G)[0] for s0, G in _groups(c, 0)])
    if op == "born_adj":
        g = zm()
        for s0, G in _groups(c, 1):
            Ds = _forward(W, s0, G, True)[1]
            for n, mu in W.back(G, W.inject(dd[s0:s0 + G])):
                g += (Ds[n] * mu[:, W.rows])[..., ph].sum(0)
        return g * W.b
    if op == "tomo":
        Wt, dv, out = W.b * pt, t["dv"].double(), []
        W2 = (-3.0 * dv / W.v) * Wt
        for s0, G in _groups(c, 3):
            D0 = _forward(W, s0, G, True)[1]
            bdv = torch.zeros(W.nz, W.NX, device=DEV, dtype=torch.float64)
            bdv[:, ph] = W.b * dv
            Dq = [D.clone() for _, _, D in W.march(G, _source_rows(W, lambda n: bdv * D0[n])) if D is not None]
            Dsc = _born_ext(W, Wt, D0, G, True)[1]
            src = lambda n: bdv * Dsc[n] + W.scatter(W2, D0[n]) + W.scatter(Wt, Dq[n])  # noqa: E731
            d = torch.zeros(G, W.nt, len(W.rx), device=DEV, dtype=torch.float64)
            for n, q, _ in W.march(G, _source_rows(W, src)):
                d[:, n] = W.record(q)
            out.append(d)
        return torch.cat(out)
    if op == "pair":
        data, I = [], zm(W.nh)
        for s0, G in _groups(c, 1):
            Ds = _forward(W, s0, G, True)[1]
            data.append(_born_ext(W, W.b * pt, Ds, G)[0])
            _ext_image(W, I, Ds, dd[s0:s0 + G])
        return torch.cat(data), I * W.b
    if op == "vp":
        groups = _groups(c, 1)
        hist = [(s0, G, _forward(W, s0, G, True)[1]) for s0, G in groups]

        def B(p):
            return torch.cat([_born_ext(W, W.b * p, Ds, G)[0] for s0, G, Ds in hist])

        def Bt(d):
            I = zm(W.nh)
            for s0, G, Ds in hist:
                _ext_image(W, I, Ds, d[s0:s0 + G])
            return I * W.b
        p = zm(W.nh)
        phi = lambda q: 0.5 * float((B(q) - dd).square().sum()) + 0.5 * eps ** 2 * float((dso * q).square().sum())  # noqa
        r = Bt(dd)
        s, rr, out = r.clone(), r.square().sum(), [0.5 * float(dd.square().sum())]
        for _ in range(c["niter"]):
            H = Bt(B(s)) + eps ** 2 * dso ** 2 * s
            a = rr / (s * H).sum()
            p, r = p + a * s, r - a * H
            rn = r.square().sum()
            s, rr = r + (rn / rr) * s, rn
            out.append(phi(p))
        return p, out
    # objective, gradient
    Wt, J, g1, I, f2 = W.b * pt, 0.0, zm(), zm(W.nh), 1.0 / W.dt ** 2
    for s0, G in _groups(c, 2.2):
        d0, D0 = _forward(W, s0, G, True)
        d1, Dsc = _born_ext(W, Wt, D0, G, op == "gradient")
        r = d0 + d1 - dd[s0:s0 + G]
        J += 0.5 * float(r.square().sum())
        if op == "objective":
            continue
        z = {}

        def second(r):
            """Drives the second adjoint field one step behind the first: yields (n, lambda^n, mu2^n)."""
            first = W.back(G, W.inject(r))
            held = {}

            def fetch(n):
                if n >= 0:
                    k, mu = next(first)
                    held[k] = mu[:, W.rows].clone()
                    z[k] = W.scatter(Wt, held[k], -1)

            def inj(n, a):     # adjoint of q^n gains (z^(n-1) - 2 z^n + z^(n+1)) / dt^2
                fetch(n - 1)
                for k, f in ((n - 1, f2), (n, -2.0 * f2), (n + 1, f2)):
                    if k in z:
                        a[:, W.rows].add_(z[k], alpha=f)
                z.pop(n + 1, None)
            for n, mu2 in W.back(G, inj):
                yield n, held.pop(n), mu2
        for n, lam, mu2 in second(r):
            g1 += (D0[n] * (lam + mu2[:, W.rows]) + Dsc[n] * lam)[..., ph].sum(0)
            W.image(I, D0[n], lam)
    J += 0.5 * eps ** 2 * float((dso * pt).square().sum())
    if op == "objective":
        return J
    return J, W.b * g1 - 3.0 * W.b / W.v * (pt * I).sum(0)
