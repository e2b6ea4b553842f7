"""Timing cases of the photoacoustic forward / adjoint library, through its Python entry points.

Each case is one call (or one differentiation step) that a reconstruction program makes again and
again: a forward record with its gradient, a batch of uneven instances, a checkpointed medium gradient,
a time-reversal image, one TV proximal map, a short multi-grid FISTA run.  Grid sizes, media, sensor
layouts and precisions are those of the package's own workloads (``synth``), its benchmark and its
tests; record lengths are shortened where a full one would take more than a second or so (the time per
step does not depend on the length).

``exact`` restates the discrete scheme in plain torch, FP64, with torch's own FFTs.
"""
import math

import numpy as np
import torch

from paper_1603_02329_gb300.api import PATBatch, PATOperator, mg_fista, tv_prox
from paper_1603_02329_gb300.autograd import pat_apply, pat_apply_batch

PML_ALPHA = 2.0
CFL = 0.3
ALPHA0, Y = 0.75, 1.5          # dB MHz^-y cm^-1
DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def _case(name, kind, shape, nt, f64=False, lossy=True, sensors="line", ns=0, pml=0, **more):
    c = dict(name=name, kind=kind, shape="x".join(map(str, shape)), nt=nt, f64=f64, lossy=lossy, sensors=sensors,
             ns=ns or shape[-1], pml=pml or max(2, min(20, min(shape) // 10)))
    c.update(more)
    return c


def listed():
    return [
        # the smallest reconstruction step the tests use: launch and barrier latency
        _case("step_2d_64", "pair", (64, 64), 120, sensors="circle", ns=48, pml=8),
        # the disc phantom in double precision, lossless: the parity workload (128^2 plus its PML)
        _case("step_2d_168_f64", "pair", (168, 168), 600, f64=True, lossy=False, sensors="circle", ns=256, pml=20),
        # the absorbing 2-D vessel workload: one objective-and-gradient evaluation, half a record
        _case("step_2d_512", "pair", (512, 512), 1000, pml=20),
        # its data generated on a 1.44 times finer grid (off-grid sensors): a forward run, ragged lines
        _case("data_2d_750", "forward", (750, 750), 400, sensors="circle", ns=512, pml=29),
        # the eight uneven 2-D instances, one batched call each way
        _case("batch_2d_uneven", "batch", (384, 384), 300, sensors="circle", ns=256, pml=20,
              sizes="192,224,256,256,288,320,320,384"),
        # time reversal: the image a reconstruction is started from
        _case("reversal_2d_256", "reversal", (256, 256), 500, pml=20),
        # the absorbing 3-D tube workloads with a planar array: one evaluation and its gradient
        _case("step_3d_128", "pair", (128, 128, 128), 200, sensors="plane", ns=4096, pml=10),
        _case("step_3d_256", "pair", (256, 256, 256), 40, sensors="plane", ns=16384, pml=10),
        # a flat 3-D slab under a top-surface array: sides that are no powers of two
        _case("step_3d_slab", "pair", (40, 160, 160), 200, sensors="plane", ns=1296, pml=4),
        # joint medium gradient (c0^2, rho0, p0) by the checkpointed sweep
        _case("medium_3d_128", "medium", (128, 128, 128), 60, sensors="plane", ns=4096, pml=10, every=20),
        # the TV proximal map of one 3-D iteration (20 inner steps)
        _case("prox_3d_256", "prox", (256, 256, 256), 0, ns=1),
        # a whole two-level multi-grid FISTA call: four iterations on noisy line-array data
        _case("mgfista_2d_256", "mgfista", (256, 256), 400, pml=20, iters=4),
    ]


def _smooth(lo, hi, step=2):
    """Multiples of ``step`` in [lo, hi] with prime factors 2, 3, 5, 7 (the transform lengths)."""
    out = []
    for n in range(lo, hi + 1):
        m = n
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1 and n % step == 0:
            out.append(n)
    return out


def _size(rng, lo, hi, step=2):
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_smooth(lo, hi, step), key=lambda n: abs(n - want))


def draw(rng):
    kind = rng.choice(("pair", "pair", "pair", "pair3", "pair3", "pair3", "forward", "batch", "reversal", "medium", "prox", "mgfista"))
    steps = lambda n, most: max(20, min(rng.randint(60, 600), int(most / n)))  # noqa: E731
    if kind == "prox":
        three = rng.random() < 0.5
        shape = tuple(_size(rng, 24, 256) for _ in range(3)) if three else tuple(_size(rng, 48, 1024) for _ in range(2))
        return _nameless(_case("", "prox", shape, 0, f64=rng.random() < 0.2, ns=1))
    if kind in ("pair3", "medium"):
        side = _size(rng, 24, 192 if kind == "pair3" else 112)
        shape = tuple(_size(rng, max(16, side // 2), min(256, 2 * side)) for _ in range(3))
        while math.prod(shape) > 3 * 2 ** 20:
            shape = tuple(_size(rng, 24, max(25, n - 2)) for n in shape)
        pml = max(2, min(shape) // 12)
        plane = max(2, min(shape[1:]) // 4)
        more = dict(every=rng.choice((5, 10, 20))) if kind == "medium" else {}
        return _nameless(_case("", "pair" if kind == "pair3" else kind, shape, steps(math.prod(shape), 4e8 if kind == "pair3" else 6e7),
                               f64=rng.random() < 0.1, lossy=rng.random() < 0.85, sensors="plane", ns=plane * plane, pml=pml, **more))
    if kind == "batch":
        sizes = sorted(_size(rng, 64, 384) for _ in range(rng.randint(2, 8)))
        return _nameless(_case("", "batch", (sizes[-1],) * 2, steps(sum(n * n for n in sizes), 1.5e8), sensors="circle",
                               ns=rng.randint(16, 256), pml=rng.randint(4, 6), sizes=",".join(map(str, sizes))))
    if kind == "mgfista":
        n = _size(rng, 64, 320, 4)
        return _nameless(_case("", "mgfista", (n, n), rng.randint(100, 400), pml=2 * rng.randint(2, max(2, n // 24)), iters=rng.randint(2, 4)))
    f64 = kind != "reversal" and rng.random() < 0.15
    n = _size(rng, 32, 384 if f64 or kind == "reversal" else 800)
    shape = (_size(rng, max(32, n // 2), n), n)
    sensors = "line" if kind == "reversal" else rng.choice(("line", "circle"))
    return _nameless(_case("", kind, shape, steps(math.prod(shape), 2e7 if f64 else 2e8), f64=f64, lossy=rng.random() < 0.85,
                           sensors=sensors, ns=shape[-1] if sensors == "line" else rng.randint(8, 512)))


def _nameless(c):
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _noise(g, shape, sigma):
    """Unit-variance white noise under a periodic Gaussian filter of ``sigma`` points."""
    w = torch.fft.fftn(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64))
    for ax, n in enumerate(shape):
        f = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
        w *= torch.exp(-2 * (math.pi * sigma * f) ** 2).reshape([-1 if a == ax else 1 for a in range(len(shape))])
    s = torch.fft.ifftn(w).real
    s -= s.mean()
    return s / s.std()


def _balls(g, shape, face=None, count=7):
    """Overlapping discs or balls of amplitude 0.5 .. 1 away from the edges, as the phantoms have them;
    with a sensor array on the plane ``face`` of the first axis they lie from just under it downwards."""
    out = torch.zeros(shape, device=DEV, dtype=torch.float64)
    u = torch.rand((count, len(shape) + 2), generator=g, device=DEV, dtype=torch.float64).tolist()
    for k, row in enumerate(u):
        r2 = 0
        for ax, n in enumerate(shape):
            at = (0.3 + 0.4 * row[ax]) * n
            if ax == 0 and face is not None:
                at = face + (0.04 + 0.6 * row[ax] * k / count) * n
            x = torch.arange(n, device=DEV, dtype=torch.float64) - at
            r2 = r2 + (x * x).reshape([-1 if a == ax else 1 for a in range(len(shape))])
        rad = (0.03 + 0.09 * row[-2]) * min(shape)
        out = torch.where(r2 <= rad * rad, torch.clamp(out, min=0.5 + 0.5 * row[-1]), out)
    return out


class _Problem:
    """One medium, sensor array, time axis and phantom, made from the seed alone."""

    def __init__(self, case, seed, shape=None):
        g = _gen(seed)
        self.shape = shape or _shape(case)
        d = len(self.shape)
        self.h = 0.0625e-3 if d == 3 else (0.1e-3 if case["sensors"] == "circle" and not case["lossy"] else 0.05e-3)
        sigma = min(8.0, min(self.shape) / 12)
        if case["lossy"]:
            self.c = 1500.0 + 100.0 * _noise(g, self.shape, sigma)
            self.rho = 1000.0 * (1.0 + 0.05 * _noise(g, self.shape, sigma))
        else:
            self.c = torch.full(self.shape, 1500.0, device=DEV, dtype=torch.float64)
            self.rho = torch.full(self.shape, 1000.0, device=DEV, dtype=torch.float64)
        self.alpha0 = ALPHA0 if case["lossy"] else 0.0
        self.pml, self.nt = int(case["pml"]), int(case["nt"])
        self.dt = CFL * self.h / float(self.c.max())
        self.dtype = torch.float64 if case["f64"] else torch.float32
        self.p0 = _balls(g, self.shape, None if case["sensors"] == "circle" else self.pml).to(self.dtype)
        self.index = self.pos = None
        ns = int(case["ns"])
        if case["sensors"] == "circle":        # off-grid points, multilinear weights
            th = 2 * math.pi * np.arange(ns) / ns
            rad = 0.33 * min(self.shape) * self.h
            self.pos = np.stack([rad * np.cos(th), rad * np.sin(th)], axis=1)
        elif d == 2:                           # a line on the first row inside the PML
            self.index = (self.pml * self.shape[1] + np.arange(ns)).astype(np.int64)
        else:                                  # a planar array on the face z = pml
            m = math.isqrt(ns)
            nz, ny, nx = self.shape
            sy, sx = max(1, ny // m), max(1, nx // m)
            ys, xs = (ny - sy * m) // 2 + sy * np.arange(m), (nx - sx * m) // 2 + sx * np.arange(m)
            self.index = ((self.pml * ny + ys[:, None]) * nx + xs[None, :]).ravel().astype(np.int64)
        self.ns = len(self.index) if self.index is not None else len(self.pos)
        # a residual: noise on top of slow variations of the record
        r = torch.randn((self.nt, self.ns), generator=g, device=DEV, dtype=torch.float64) if self.nt else torch.zeros((1, 1))
        self.h_res = (0.1 * (r + torch.cumsum(r, 0) / math.sqrt(max(1, self.nt)))).to(self.dtype)

    def operator(self):
        d = len(self.shape)
        return PATOperator(self.shape, (self.h,) * d, (self.pml,) * d, PML_ALPHA, self.c.cpu().numpy(), self.rho.cpu().numpy(),
                           self.alpha0, Y, self.dt, self.nt, sensor_pos=self.pos, sensor_index=self.index,
                           precision="f64" if self.dtype == torch.float64 else "f32")


def _noisy_data(pb, seed):
    """The phantom's record with noise at 40 dB, as a measurement gives it."""
    d = _Exact(pb).forward(pb.p0.double())
    sigma = d.square().mean().sqrt() * 10 ** (-40 / 20)
    return (d + sigma * torch.randn(d.shape, generator=_gen(seed + 7), device=DEV, dtype=torch.float64)).to(pb.dtype).contiguous()


def _two_digits(v):
    """``v`` rounded up to two digits: the Lipschitz constant a program notes down once per plan."""
    e = 10.0 ** (math.floor(math.log10(v)) - 1)
    return math.ceil(v / e) * e


def prepare(case, seed):
    kind, shape = case["kind"], _shape(case)
    if kind == "prox":
        z = _balls(_gen(seed), shape) + 0.1 * torch.randn(shape, generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
        return dict(kind=kind, z=z.to(torch.float64 if case["f64"] else torch.float32).contiguous(), weight=0.05)
    if kind == "batch":
        pbs = [_Problem(case, seed * 16 + i, (n, n)) for i, n in enumerate(int(v) for v in case["sizes"].split(","))]
        ops = [pb.operator() for pb in pbs]
        return dict(kind=kind, ops=ops, batch=PATBatch(ops), p0=[pb.p0.requires_grad_(True) for pb in pbs],
                    res=[pb.h_res for pb in pbs])
    pb = _Problem(case, seed)
    op = pb.operator()
    if kind == "reversal":
        return dict(kind=kind, op=op, data=_noisy_data(pb, seed))
    if kind == "mgfista":
        coarse = op.coarse()
        v0 = torch.rand(shape, generator=_gen(seed + 3), device=DEV, dtype=torch.float64).to(pb.dtype)
        v0c = torch.rand(coarse.shape, generator=_gen(seed + 4), device=DEV, dtype=torch.float64).to(pb.dtype)
        return dict(kind=kind, op=op, coarse=coarse, data=_noisy_data(pb, seed), x0=torch.zeros_like(pb.p0), iters=int(case["iters"]),
                    L=_two_digits(1.2 * op.power_iteration(v0, 6)), Lc=_two_digits(1.2 * coarse.power_iteration(v0c, 6)))
    return dict(kind=kind, op=op, p0=pb.p0.requires_grad_(kind == "pair"), res=pb.h_res, every=int(case.get("every", 0)))


def run(state):
    kind = state["kind"]
    if kind == "pair":
        data = pat_apply(state["op"], state["p0"])
        grad, = torch.autograd.grad(data, state["p0"], state["res"])
        return {"data": data, "grad": grad}
    if kind == "forward":
        return {"data": state["op"].forward(state["p0"])}
    if kind == "batch":
        data = pat_apply_batch(state["ops"], state["p0"], state["batch"])
        return {"data": list(data), "grad": list(torch.autograd.grad(data, state["p0"], state["res"]))}
    if kind == "reversal":
        return {"image": state["op"].time_reversal(state["data"])}
    if kind == "medium":
        rho, c2, p0 = state["op"].gradient_medium(state["p0"], state["res"], state["every"])
        return {"rho": rho, "c2": c2, "p0": p0}
    if kind == "prox":
        return {"x": tv_prox(state["z"], state["weight"])}
    x, report, _ = mg_fista(state["op"], state["coarse"], state["data"], state["x0"], state["L"], state["Lc"], lam=1e-3,
                            max_iter=state["iters"], eps_d=0.0)
    return {"x": x, "F": report["F"], "RES": report["RES"], "solves": report["fwd_solves"] + report["adj_solves"]}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _solve_work(shape, nt, ns, f64, lossy):
    """One solve: per step the split state read and written once and the medium read once (where the
    state of a small grid can stay on the chip less would do; it is counted all the same), and the real
    transforms of the three spectral operations."""
    d, n, w = len(shape), math.prod(shape), 8 if f64 else 4
    fields = 2 * (2 * d + 1) + (4 if lossy else 2)           # u_xi, rho_xi, p both ways; c0^2, rho0, tau, eta
    transforms = (1 + d) + 2 * d + (4 if lossy else 0)
    return dict(bytes=nt * (fields * n + ns) * w, flops=nt * n * (transforms * 2.5 * math.log2(n) + 12 * d + 10))


def work(case):
    kind, shape, f64 = case["kind"], _shape(case), case["f64"]
    n, d = math.prod(shape), len(shape)
    w = 8 if f64 else 4
    if kind == "prox":    # per inner step: z and the last two duals read, the new one written
        return dict(bytes=20 * (1 + 3 * d) * n * w, flops=20 * n * 12 * d)
    shapes = [shape] if kind != "batch" else [(int(v),) * 2 for v in case["sizes"].split(",")]
    one = [_solve_work(s, case["nt"], case["ns"], f64, case["lossy"]) for s in shapes]
    # forward and adjoint; the medium sweep recomputes the forward once; an iteration is about a pair
    times = dict(forward=1, reversal=1, pair=2, batch=2, medium=3).get(kind) or 2 * int(case["iters"]) + 1
    return {k: times * sum(o[k] for o in one) for k in ("bytes", "flops")}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------------
class _Exact:
    """The discrete scheme of one problem: split-field PML, staggered k-space derivatives with the
    sinc correction, power-law absorption by two fractional Laplacians, multilinear sensors."""

    def __init__(self, pb):
        shape, d = pb.shape, len(pb.shape)
        self.pb, self.shape, self.d, self.dt, self.nt, self.lossy = pb, shape, d, pb.dt, pb.nt, pb.alpha0 != 0
        cref = float(pb.c.max())
        self.c2, self.rho = pb.c ** 2, pb.rho
        axes = [d - 1 - a for a in range(d)]                     # numpy axis of x, y, z
        view = lambda v, ax: torch.as_tensor(v, device=DEV).reshape([-1 if a == ax else 1 for a in range(d)])  # noqa: E731
        self.b, self.a, self.au, ks = [], [], [], []
        for xi, ax in enumerate(axes):
            n = shape[ax]
            self.b.append(2.0 / (pb.rho + torch.roll(pb.rho, -1, ax)))
            pos = np.arange(n, dtype=np.float64)
            sig = lambda p: PML_ALPHA * cref / pb.h * (np.maximum(np.maximum(pb.pml - p, p - (n - 1 - pb.pml)), 0) / pb.pml) ** 4  # noqa: B023,E731
            self.a.append(view(np.exp(-sig(pos) * pb.dt / 2), ax))
            self.au.append(view(np.exp(-sig(pos + 0.5) * pb.dt / 2), ax))
            m = np.arange(n // 2 + 1 if xi == 0 else n)
            ks.append(view(2 * np.pi * np.where(m > n // 2, m - n, m) / (n * pb.h), ax))
        k2 = sum(k * k for k in ks)
        kap = torch.sinc(cref * pb.dt / 2 / math.pi * torch.sqrt(k2))
        self.dp = [1j * k * torch.exp(0.5j * k * pb.h) * kap for k in ks]
        self.dm = [1j * k * torch.exp(-0.5j * k * pb.h) * kap for k in ks]
        if self.lossy:
            pw = lambda s: torch.where(k2 > 0, torch.where(k2 > 0, k2, 1.0) ** (s / 2), 0.0)  # noqa: E731
            self.l1, self.l2 = pw(Y - 2), pw(Y - 1)
            self.kmag = torch.sqrt(k2)
            a0 = pb.alpha0 * 100.0 / (20 * math.log10(math.e)) * (2 * math.pi * 1e6) ** (-Y)
            self.ct = self.c2 * (-2 * a0 * pb.c ** (Y - 1))
            self.ce = self.c2 * (2 * a0 * pb.c ** Y * math.tan(math.pi * Y / 2))
        if pb.index is not None:
            self.at, self.wt = torch.as_tensor(pb.index, device=DEV)[None], torch.ones((1, 1), device=DEV, dtype=torch.float64)
        else:
            f = pb.pos / pb.h + np.array([shape[1] // 2, shape[0] // 2])
            i, t = np.floor(f).astype(np.int64), f - np.floor(f)
            at, wt = [], []
            for cy in (0, 1):
                for cx in (0, 1):
                    at.append((i[:, 1] + cy) * shape[1] + i[:, 0] + cx)
                    wt.append((t[:, 0] if cx else 1 - t[:, 0]) * (t[:, 1] if cy else 1 - t[:, 1]))
            self.at, self.wt = torch.as_tensor(np.stack(at), device=DEV), torch.as_tensor(np.stack(wt), device=DEV)

    def fft(self, f):
        return torch.fft.fftn(torch.fft.rfft(f, dim=-1), dim=tuple(range(self.d - 1)))

    def ifft(self, s):
        s = torch.fft.ifftn(s, dim=tuple(range(self.d - 1)))
        s.imag[..., 0] = 0
        s.imag[..., -1] = 0
        return torch.fft.irfft(s, n=self.shape[-1], dim=-1)

    def sample(self, p):
        return (p.reshape(-1)[self.at] * self.wt).sum(0)

    def spread(self, h):
        p = torch.zeros(math.prod(self.shape), device=DEV, dtype=torch.float64)
        p.index_add_(0, self.at.reshape(-1), (self.wt * h.double()[None]).reshape(-1))
        return p.reshape(self.shape)

    def steps(self, p, u, rh, first=None, l1=None, tau=1.0, enforce=None, keep=None):
        """The time steps from (p, u, rh); yields the pressure of each level after the first."""
        l1 = self.l1 if l1 is None and self.lossy else l1
        for n in range(self.nt - 1):
            pk = self.fft(p)
            g = [self.ifft(m * pk) for m in self.dp]
            if n == 0 and first:
                u = [0.5 * self.dt * b * gi for b, gi in zip(self.b, g)]
            u = [au * (au * ui - self.dt * b * gi) for au, ui, b, gi in zip(self.au, u, self.b, g)]
            e = [self.ifft(m * self.fft(ui)) for m, ui in zip(self.dm, u)]
            rh = [a * (a * r - self.dt * self.rho * ei) for a, r, ei in zip(self.a, rh, e)]
            r = sum(rh)
            q = r
            p = self.c2 * r
            if self.lossy:
                ld = self.ifft(l1 * self.fft(self.rho * sum(e)))
                lr = self.ifft(self.l2 * self.fft(r))
                p = p + tau * self.ct * ld - self.ce * lr
                q = r + ((Y + 1) / 2 * self.ct * ld - (Y + 2) / 2 * self.ce * lr) / self.c2
            if enforce is not None:
                p, rh = enforce(n + 1, p, rh)
            if keep is not None:
                keep.append((g, e, q))
            yield p

    def forward(self, p0, keep=None):
        rows = [self.sample(p0)]
        for p in self.steps(p0, None, [p0 / (self.d * self.c2)] * self.d, first=True, keep=keep):
            rows.append(self.sample(p))
        return torch.stack(rows)

    def adjoint(self, h, kept=None, p0=None):
        """H^T h; with the forward's kept fields also the products for c0^2 and rho0."""
        dt, d = self.dt, self.d
        p = self.spread(h[self.nt - 1])
        zero = torch.zeros(self.shape, device=DEV, dtype=torch.float64)
        u, rh = [zero] * d, [zero] * d
        gc, gr, gb = zero.clone(), zero.clone(), [zero.clone() for _ in range(d)]
        for n in range(self.nt - 2, -1, -1):
            g, e, q = kept[n] if kept else (None, None, None)
            if kept:
                gc += p * q
            rbar, ddbar = self.c2 * p, zero
            if self.lossy:
                ddbar = self.ifft(self.l1 * self.fft(self.ct * p))
                rbar = rbar - self.ifft(self.l2 * self.fft(self.ce * p))
            rh = [r + rbar for r in rh]
            eb = [self.rho * ddbar - dt * self.rho * a * r for a, r in zip(self.a, rh)]
            if kept:
                gr += sum(ei * (ddbar - dt * a * r) for ei, a, r in zip(e, self.a, rh))
            rh = [a * a * r for a, r in zip(self.a, rh)]
            u = [ui - self.ifft(m * self.fft(ei)) for ui, m, ei in zip(u, self.dp, eb)]
            gbar = [-dt * b * au * ui for b, au, ui in zip(self.b, self.au, u)]
            if kept:
                for k in range(d):
                    gb[k] += u[k] * (-dt * self.au[k] * g[k])
            u = [au * au * ui for au, ui in zip(self.au, u)]
            if n == 0:
                gbar = [gi + 0.5 * dt * b * ui for gi, b, ui in zip(gbar, self.b, u)]
                if kept:
                    for k in range(d):
                        gb[k] += u[k] * 0.5 * dt * g[k]
            acc = sum(m * self.fft(gi) for m, gi in zip(self.dm, gbar))
            p = self.spread(h[n]) - self.ifft(acc)
        s = sum(rh)
        gp = p + s / (d * self.c2)
        if not kept:
            return gp
        gc -= s * p0 / (d * self.c2 ** 2)
        for k in range(d):
            v = gb[k] * (-0.5 * self.b[k] ** 2)
            gr += v + torch.roll(v, 1, d - 1 - k)
        return gr, gc, gp

    def reversal(self, data, k_cut=0.5):
        """The time-reversal image: reversed data enforced at the (on-grid) sensors, the absorption
        term reversed in sign and cut by a Blackman window at ``k_cut`` of the Nyquist radius."""
        data = data.double()
        at, d = self.at[0], self.d
        c2s = self.c2.reshape(-1)[at]

        def put(n, p, rh):
            row = data[self.nt - 1 - n]
            p, rh = p.clone().reshape(-1), [r.clone().reshape(-1) for r in rh]
            p[at] = row
            for r in rh:
                r[at] = row / (d * c2s)
            return p.reshape(self.shape), [r.reshape(self.shape) for r in rh]

        l1 = None
        if self.lossy:
            q = self.kmag / (k_cut * math.pi / self.pb.h)
            win = torch.where(q < 1, 0.42 + 0.5 * torch.cos(math.pi * q) + 0.08 * torch.cos(2 * math.pi * q), 0.0)
            l1 = -win * self.l1
        p = torch.zeros(self.shape, device=DEV, dtype=torch.float64).reshape(-1)
        p[at] = data[self.nt - 1]
        p = p.reshape(self.shape)
        zero = torch.zeros_like(p)
        for p in self.steps(p, [zero] * d, [p / (d * self.c2)] * d, l1=l1, enforce=put):
            pass
        return p


def _exact_prox(z, weight, n_inner=20):
    """argmin weight TV(x) + [x >= 0] + 1/2 |x - z|^2 by the dual fast gradient projection."""
    z, d = z.double(), z.dim()
    weight, step, t = float(weight), 1.0 / (4 * z.dim() * float(weight)), 1.0

    def grad(x):
        out = []
        for ax in range(d):
            g = torch.zeros_like(x)
            g.narrow(ax, 0, x.shape[ax] - 1).copy_(x.narrow(ax, 1, x.shape[ax] - 1) - x.narrow(ax, 0, x.shape[ax] - 1))
            out.append(g)
        return out

    def primal(q):
        v = z.clone()
        for ax in range(d):
            n = z.shape[ax]
            v.narrow(ax, 1, n - 1).sub_(weight * q[ax].narrow(ax, 0, n - 1))
            v.narrow(ax, 0, n - 1).add_(weight * q[ax].narrow(ax, 0, n - 1))
        return v.clamp_(min=0)

    q = [torch.zeros_like(z) for _ in range(d)]
    r = q
    for _ in range(n_inner):
        new = [ri + step * gi for ri, gi in zip(r, grad(primal(r)))]
        norm = torch.sqrt(sum(v * v for v in new)).clamp_(min=1.0)
        new = [v / norm for v in new]
        tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
        r = [v + (t - 1) / tn * (v - o) for v, o in zip(new, q)]
        q, t = new, tn
    return primal(q)


def exact(case, seed):
    kind = case["kind"]
    if kind == "mgfista":       # a whole optimisation: some hundred solves
        return None
    if kind == "prox":
        s = prepare(case, seed)
        return {"x": _exact_prox(s["z"], s["weight"])}
    if kind == "batch":
        data, grad = [], []
        for i, n in enumerate(int(v) for v in case["sizes"].split(",")):
            pb = _Problem(case, seed * 16 + i, (n, n))
            ex = _Exact(pb)
            data.append(ex.forward(pb.p0.double()))
            grad.append(ex.adjoint(pb.h_res.double()))
        return {"data": data, "grad": grad}
    pb = _Problem(case, seed)
    ex = _Exact(pb)
    if kind == "reversal":
        return {"image": ex.reversal(_noisy_data(pb, seed))}
    p0, res = pb.p0.double(), pb.h_res.double()
    if kind == "medium":
        kept = []
        ex.forward(p0, kept)
        rho, c2, gp = ex.adjoint(res, kept, p0)
        return {"rho": rho, "c2": c2, "p0": gp}
    data = ex.forward(p0)
    return {"data": data} if kind == "forward" else {"data": data, "grad": ex.adjoint(res)}
