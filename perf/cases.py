"""Performance cases of the PSD solver: what a user's program calls, from one
residual on a small grid to a whole sixth-order solve on 256^3 cells.

Every case goes through the public entry points (``Solver``, ``Batch``,
``psd_solve_autograd``).  ``prepare`` makes what a program holds before the
call (fields on the GPU and the handle), ``run`` is one call, ``exact`` is the
same result by plain torch operations in 64 bits: the stencils as rolls, the
solves by Newton's method with conjugate gradients.
"""

import math
import os

# the batch's documented setting: hardware queues for its concurrent instances
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import torch  # noqa: E402

from paper_1607_01475_gb300 import PSD_FP64, PSD_MIXED, Batch, Solver  # noqa: E402
from paper_1607_01475_gb300.autograd import psd_solve_autograd  # noqa: E402

TWO_PI = 2.0 * math.pi
PRECISION = {"fp64": PSD_FP64, "mixed": PSD_MIXED}


def _case(name, kind, shape, **opts):
    shape = list(shape) + [0] * (3 - len(shape))
    base = dict(kind=kind, n0=shape[0], n1=shape[1], n2=shape[2], order=4, precision="fp64", p=4.0, s=0.1,
                eps=0.05, lam=0.0, tol=0.0)
    base.update(opts)
    if name:
        base["name"] = name
    return base


def listed():
    return [
        # one residual of a small 2D field: the smallest call, as a program's
        # own convergence check or a diagnostic makes it
        _case("residual_2d_64", "residual", (64, 64), s=0.01, eps=0.1),
        # one preconditioner solve on a non-cubic box, FP64 (a user's own
        # iteration around the FFT solve)
        _case("precond_64x256x128", "precond", (64, 256, 128)),
        # plain FP64 solve of a small 2D grid: launches and latency
        _case("solve_2d_64_fp64", "solve", (64, 64), s=0.01, eps=0.1),
        # thin-film shaped 2D solve, mixed precision
        _case("solve_2d_1024_mixed", "solve", (1024, 1024), precision="mixed", tol=1e-10),
        # thin-film shaped 3D solve in both precisions
        _case("solve_3d_128_fp64", "solve", (128, 128, 128)),
        _case("solve_3d_128_mixed", "solve", (128, 128, 128), precision="mixed"),
        # the sixth-order system on 256^3 in both precisions: the benchmark
        _case("solve6_3d_256_fp64", "solve", (256, 256, 256), order=6, s=0.05, eps=0.1, lam=1.0),
        _case("solve6_3d_256_mixed", "solve", (256, 256, 256), order=6, s=0.05, eps=0.1, lam=1.0,
              precision="mixed"),
        # 96 uneven 2D instances (64^2 .. 1024^2, p = 3 and 4), one batch call
        _case("batch_96_mixed", "batch", (96,), precision="mixed"),
        # forward and backward of the differentiable solve
        _case("grad_3d_128_mixed", "grad", (128, 128, 128), precision="mixed"),
        # time loops: thin-film epitaxy (mixed) and square phase field crystal
        # (FP64), 10 steps a call
        _case("thinfilm_2d_512_mixed", "thinfilm", (512, 512), precision="mixed", eps=0.1, s=0.0),
        _case("spfc_2d_256_fp64", "spfc", (256, 256), order=6, s=0.01, eps=1.0, lam=0.5),
    ]


def _draw_shape(rng, dim, lo, hi, cells):
    while True:
        shape = [2 ** rng.randint(lo, hi) for _ in range(dim)]
        if math.prod(shape) <= cells:
            return shape


def draw(rng):
    kind = rng.choice(["residual", "precond", "solve", "solve", "solve", "grad", "thinfilm", "spfc", "batch"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "batch":
        return _case("", kind, (rng.randint(2, 96),), precision="mixed")
    if kind in ("thinfilm", "spfc"):
        n = 2 ** rng.randint(5, 10)  # square boxes, as the runs of the paper
        if kind == "thinfilm":
            return _case("", kind, (n, n), precision=precision, p=rng.choice([4.0, 6.0]), eps=0.1, s=0.0)
        return _case("", kind, (n, n), order=6, precision=precision, s=0.01, eps=1.0, lam=0.5)
    dim = rng.choice([2, 3])
    s = 10.0 ** rng.uniform(-2.0, -1.0)
    eps = rng.uniform(0.05, 0.1)
    if kind in ("residual", "precond"):
        # any exponent, grids from 8 to 1024 per axis
        shape = _draw_shape(rng, dim, 3, 10, 1 << 24)
        return _case("", kind, shape, order=rng.choice([4, 6]), precision=precision, lam=1.0,
                     p=rng.choice([3.0, 4.0, 5.0, 6.0]) if kind == "residual" else 4.0, s=s, eps=eps)
    if kind == "grad":
        shape = _draw_shape(rng, dim, 4, 9, 1 << 21)
        return _case("", kind, shape, precision=precision, s=min(s, _largest_s(shape, eps)), eps=eps)
    p = rng.choice([3.0, 4.0, 4.0])
    order = rng.choice([4, 6])
    cells = 1 << 24 if p == 4.0 else 1 << 18
    shape = _draw_shape(rng, dim, 3 if dim == 3 else 4, 10 if dim == 2 else 8, cells)
    return _case("", "solve", shape, order=order, precision=precision, p=p,
                 s=min(s, _largest_s(shape, eps)), eps=eps, lam=1.0)


# ------------------------------------------------------------------- inputs


def _shape(case):
    return tuple(n for n in (case["n0"], case["n1"], case["n2"]) if n)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed), torch.Generator().manual_seed(seed + 1)


def _fourier(shape, h, K, cpu, amp=1.0, nmodes=32):
    """32 random Fourier modes with |k| <= K of the box, N(0,1) amplitudes
    over 1 + |k|^2 (the right-hand sides of the benchmark workloads)."""
    dim = len(shape)
    ks = []
    while len(ks) < nmodes:
        k = (torch.rand(dim, generator=cpu, dtype=torch.float64) * (2 * K + 1)).floor() - K
        if 0 < float((k * k).sum()) <= K * K:
            ks.append(k)
    k = torch.stack(ks)
    w = torch.randn(nmodes, 2, generator=cpu, dtype=torch.float64) / (1.0 + (k * k).sum(1))[:, None]
    w = torch.complex(w[:, 0], -w[:, 1]).cuda()
    out = None
    for a, n in enumerate(shape):
        x = (torch.arange(n, dtype=torch.float64) + 0.5) / n
        e = torch.exp(1j * TWO_PI * k[:, a, None] * x).cuda()
        if out is None:
            out = w[:, None] * e
        elif a < dim - 1:
            out = (out[:, :, None] * e[:, None, :]).flatten(1)
        else:
            left = torch.cat([out.real, -out.imag]).T.contiguous()
            out = left @ torch.cat([e.real, e.imag])
    return (amp * out).reshape(shape).contiguous()


def _wave2(shape, h):
    """|k|^2 of the box's angular wavenumbers, half spectrum."""
    total = None
    for a, n in enumerate(shape):
        f = torch.fft.rfftfreq if a == len(shape) - 1 else torch.fft.fftfreq
        q = (TWO_PI * f(n, d=h, dtype=torch.float64, device="cuda")) ** 2
        q = q.reshape([-1 if b == a else 1 for b in range(len(shape))])
        total = q if total is None else total + q
    return total


def _phase_field_rhs(shape, h, s, gpu):
    """phi - s Delta phi of a smoothed uniform(-0.1, 0.1) phase field."""
    phi = 0.2 * torch.rand(shape, generator=gpu, dtype=torch.float64, device="cuda") - 0.1
    k2 = _wave2(shape, h)
    spec = torch.fft.rfftn(phi) * torch.exp(-k2 / 64.0) * (1.0 + s * k2)
    return torch.fft.irfftn(spec, s=shape).contiguous()


def _spacing(case, shape):
    if case["kind"] == "thinfilm":
        return 3.2 / shape[-1]
    if case["kind"] == "spfc":
        return 100.0 / shape[-1]
    return TWO_PI / max(shape)


def _time_step(case, h):
    return 0.1 * h * h if case["kind"] == "thinfilm" else case["s"]


def _tolerance(h, f):
    """Residual tolerance of a solve: 1e-10, relative to small right-hand sides."""
    return 1e-10 * min(1.0, math.sqrt(h ** f.dim()) * float(f.norm()))


def _largest_s(shape, eps):
    """The largest s <= 0.1 for which FP64 rounding of s eps^2 Delta_h^2 u
    stays below a residual of 1e-10: on fine grids s is time-step small."""
    h = TWO_PI / max(shape)
    return min(0.1, 1.8e3 * h ** 4 / eps ** 2)


def _fields(case, seed):
    """The input fields of a case (all kinds but the batch)."""
    shape = _shape(case)
    h = _spacing(case, shape)
    gpu, cpu = _gen(seed)
    kind = case["kind"]
    new = {"shape": shape, "h": h, "s": _time_step(case, h)}
    if kind == "residual":
        # an iterate with grid-scale random data (the initial data of the
        # phase-field runs) on top of a smooth field
        noise = 0.1 * torch.rand(shape, generator=gpu, dtype=torch.float64, device="cuda") - 0.05
        new["u"] = _fourier(shape, h, 6, cpu) + noise
        new["f"] = _fourier(shape, h, 8, cpu)
        if case["order"] == 6:
            new["g"] = _fourier(shape, h, 8, cpu)
    elif kind == "precond":
        r = torch.randn(shape, generator=gpu, dtype=torch.float64, device="cuda")
        new["r"] = r.float() if case["precision"] == "mixed" else r
    elif kind == "solve" and case["order"] == 6:
        new["f"] = _fourier(shape, h, 16, cpu)
        new["g"] = _fourier(shape, h, 16, cpu)
        new["u0"] = torch.full(shape, float(new["g"].mean()), dtype=torch.float64, device="cuda")
    elif kind in ("solve", "grad"):
        new["f"] = _fourier(shape, h, 8, cpu) if math.prod(shape) <= 1 << 13 else _phase_field_rhs(shape, h, new["s"], gpu)
        new["u0"] = torch.zeros(shape, dtype=torch.float64, device="cuda")
        if kind == "grad":
            new["target"] = _fourier(shape, h, 4, cpu, amp=0.05)
    elif kind == "thinfilm":
        # the analytic initial data of the paper's thin-film test, its origin moved
        x = (torch.arange(shape[-1], dtype=torch.float64, device="cuda") + 0.5) * h
        dx, dy = (3.2 * torch.rand(2, generator=cpu, dtype=torch.float64)).tolist()
        x, y, w = x[None, :] + dx, x[:, None] + dy, TWO_PI / 3.2
        new["u0"] = (0.1 * torch.sin(w * x) ** 2 * torch.sin(2 * w * (y - 1.4))
                     - 0.1 * torch.cos(w * (x - 2.0)) * torch.sin(w * y)).contiguous()
    else:  # spfc: random data around a constant state
        new["u0"] = 0.2 + 0.1 * torch.rand(shape, generator=gpu, dtype=torch.float64, device="cuda") - 0.05
    return new


def _batch_instances(case, seed):
    """Uneven 2D instances shaped like the batch workload: 64^2 .. 1024^2, s
    up to 0.1, eps in [0.05, 0.2], p = 3 or 4."""
    gpu, cpu = _gen(seed)
    out = []
    for i in range(case["n0"]):
        # the mix of sizes and parameters is the case's, the fields are the seed's
        v = torch.rand(4, generator=torch.Generator().manual_seed(1000 + i), dtype=torch.float64).tolist()
        n = 2 ** (6 + int(5 * v[0]))
        h = TWO_PI / n
        eps, p = 0.05 + 0.15 * v[2], 3.0 if v[3] < 0.5 else 4.0
        s = min(10.0 ** (-3.0 + 2.0 * v[1]), _largest_s((n, n), eps))
        f = _fourier((n, n), h, 8, cpu)
        out.append(dict(shape=(n, n), h=h, p=p, s=s, eps=eps, f=f, tol=_tolerance(h, f)))
    return out


STEPS = 10  # time steps per call of the time loops


def prepare(case, seed):
    if case["kind"] == "batch":
        inst = _batch_instances(case, seed)
        batch = Batch([dict(order=4, shape=i["shape"], h=i["h"], p=i["p"], s=i["s"], eps=i["eps"],
                            precision=PRECISION[case["precision"]], tol=i["tol"], max_outer=60) for i in inst])
        # the solutions of one grid size side by side
        out, us = {}, []
        for n in sorted({i["shape"][0] for i in inst}):
            out[n] = torch.zeros((sum(i["shape"][0] == n for i in inst), n, n), dtype=torch.float64, device="cuda")
        seen = dict.fromkeys(out, 0)
        for i in inst:
            n = i["shape"][0]
            us.append(out[n][seen[n]])
            seen[n] += 1
        return dict(kind="batch", batch=batch, f=[i["f"] for i in inst], u=us, out=out)
    st = _fields(case, seed)
    st["kind"] = case["kind"]
    kind = case["kind"]
    if kind == "grad":
        st["f"].requires_grad_()
        st["st"] = torch.tensor(st["s"], dtype=torch.float64, device="cuda", requires_grad=True)
        st["opts"] = dict(h=st["h"], p=case["p"], eps=case["eps"], precision=PRECISION[case["precision"]],
                          tol=_tolerance(st["h"], st["f"].detach()))
        return st
    tol = 1e-11 if kind == "thinfilm" else 1e-10
    if kind == "solve":
        tol = max(_tolerance(st["h"], st["f"]), case["tol"])
    st["solver"] = Solver(case["order"], st["shape"], st["h"], case["p"], st["s"], case["eps"], case["lam"],
                          precision=PRECISION[case["precision"]], tol=tol)
    if kind == "solve" and case["precision"] == "mixed":
        st["solver"].autotune()
    if kind in ("solve", "thinfilm", "spfc"):
        st["u"] = torch.empty_like(st["u0"])
    elif kind == "residual":
        st["r"] = torch.empty_like(st["u"])
    else:
        st["d"] = torch.empty_like(st["r"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "residual":
        l2, linf = st["solver"].residual(st["u"], st["f"], st.get("g"), st["r"])
        return {"r": st["r"], "l2": l2, "linf": linf}
    if kind == "precond":
        if st["r"].dtype == torch.float32:
            st["solver"].precond_solve_f32(st["r"], st["d"])
        else:
            st["solver"].precond_solve(st["r"], st["d"])
        return st["d"]
    if kind == "batch":
        for u in st["out"].values():
            u.zero_()
        st["batch"].solve(st["f"], st["u"])
        return {str(n): u for n, u in st["out"].items()}
    if kind == "grad":
        u = psd_solve_autograd(st["f"], st["st"], **st["opts"])
        loss = 0.5 * st["h"] ** u.dim() * ((u - st["target"]) ** 2).sum()
        gf, gs = torch.autograd.grad(loss, (st["f"], st["st"]))
        return {"u": u.detach(), "grad_f": gf, "grad_s": gs}
    st["u"].copy_(st["u0"])
    if kind == "solve":
        st["solver"].solve(st["f"], st["u"], st.get("g"))
    elif kind == "thinfilm":
        st["solver"].thinfilm_steps(st["u"], STEPS)
    else:
        st["solver"].spfc_steps(st["u"], 2.0, STEPS)
    return st["u"]


# Work: fields read and written once; a solve counts the arithmetic of the
# iterations that its linear rate takes to the tolerance (about 30 here).
_ITERATIONS = {"residual": 0, "precond": 0, "solve": 30, "grad": 60, "thinfilm": 3 * STEPS, "spfc": 5 * STEPS}


def work(case):
    if case["kind"] == "batch":
        cells = sum(i["shape"][0] ** 2 for i in _batch_sizes(case))
        return {"bytes": 24.0 * cells, "flops": 30.0 * cells * (60 + 4 * 2.5 * 16)}
    shape = _shape(case)
    n = math.prod(shape)
    size = 4 if case["kind"] == "precond" and case["precision"] == "mixed" else 8
    fields = {"residual": 3, "precond": 2, "solve": 3, "grad": 4, "thinfilm": 2, "spfc": 2}[case["kind"]]
    fields += 1 if case["order"] == 6 and case["kind"] in ("residual", "solve") else 0
    transforms = 2 * 2.5 * math.log2(n)  # there and back, real data
    stencils = 60 if len(shape) == 2 else 110  # residual and line search
    if case["kind"] == "residual":
        flops = n * (stencils * 0.6 + (transforms if case["order"] == 6 else 0))
    elif case["kind"] == "precond":
        flops = n * (transforms + 8)
    else:
        flops = _ITERATIONS[case["kind"]] * n * (stencils + transforms + 16)
    return {"bytes": float(fields * size * n), "flops": float(flops)}


def _batch_sizes(case):
    out = []
    for i in range(case["n0"]):
        v = torch.rand(4, generator=torch.Generator().manual_seed(1000 + i), dtype=torch.float64).tolist()
        out.append(dict(shape=(2 ** (6 + int(5 * v[0])),) * 2))
    return out


# ------------------------------------------------ the same results in plain torch


class _Plain:
    """N_h, its derivative and the Newton solve on one periodic grid (FP64)."""

    def __init__(self, order, shape, h, p, s, eps, lam):
        self.order, self.shape, self.h, self.p, self.s, self.eps, self.lam = order, shape, h, p, s, eps, lam
        self.dim = len(shape)
        mu = None
        for a, n in enumerate(shape):
            m = n // 2 + 1 if a == self.dim - 1 else n
            k = torch.arange(m, dtype=torch.float64, device="cuda")
            q = (4.0 / h ** 2 * torch.sin(math.pi * k / n) ** 2).reshape([-1 if b == a else 1 for b in range(self.dim)])
            mu = q if mu is None else mu + q
        self.inv_mu = torch.where(mu > 0, 1.0 / torch.where(mu > 0, mu, 1.0), 0.0)
        sym = s * mu + s * eps ** 2 * mu ** 2
        sym = 1.0 + sym if order == 4 else s * lam + sym + self.inv_mu
        self.inv_sym = 1.0 / sym
        if order == 6:
            self.inv_sym = torch.where(mu > 0, self.inv_sym, 0.0)
        self.cu = 1.0 if order == 4 else s * lam

    def spectral(self, x, sym):
        return torch.fft.irfftn(torch.fft.rfftn(x) * sym, s=self.shape)

    def grad(self, u):
        """Vertex gradients: difference along one axis, averages along the others."""
        out = []
        for a in range(self.dim):
            g = u
            for b in range(self.dim):
                up = torch.roll(g, -1, b)
                g = (up - g) / self.h if a == b else 0.5 * (up + g)
            out.append(g)
        return out

    def div(self, F):
        out = 0.0
        for a in range(self.dim):
            g = F[a]
            for b in range(self.dim):
                dn = torch.roll(g, 1, b)
                g = (g - dn) / self.h if a == b else 0.5 * (g + dn)
            out = out + g
        return out

    def lap(self, u):
        out = -2.0 * self.dim * u
        for a in range(self.dim):
            out = out + (torch.roll(u, 1, a) + torch.roll(u, -1, a))
        return out / self.h ** 2

    def linear(self, u):
        out = self.cu * u + self.s * self.eps ** 2 * self.lap(self.lap(u))
        return out

    def factor(self, a2, power):
        return a2 if power == 1.0 else torch.where(a2 > 0, a2, 1.0) ** power * (a2 > 0) if power != 0 else 1.0

    def op(self, u, g=None):
        """N_h[u] (order 6: with T_h[u - g])."""
        G = self.grad(u)
        w = self.factor(sum(x * x for x in G), 0.5 * self.p - 1.0)
        out = self.linear(u) - self.s * self.div([w * x for x in G])
        return out if self.order == 4 else out + self.spectral(u - g, self.inv_mu)

    def residual(self, u, f, g=None):
        r = f - self.op(u, g)
        return r if self.order == 4 else r - r.mean()

    def hess(self, G):
        a2 = sum(x * x for x in G)
        w0 = self.factor(a2, 0.5 * self.p - 1.0)
        w1 = (self.p - 2.0) * (1.0 if self.p == 4.0 else self.factor(a2, 0.5 * self.p - 2.0))

        def apply(v):
            E = self.grad(v)
            ae = w1 * sum(x * y for x, y in zip(G, E))
            out = self.linear(v) - self.s * self.div([w0 * e + ae * x for x, e in zip(G, E)])
            return out if self.order == 4 else out + self.spectral(v, self.inv_mu)

        return apply

    def cg(self, H, b, rel, limit=400):
        x, r = torch.zeros_like(b), b
        z = self.spectral(r, self.inv_sym)
        p, rz, stop = z, (r * z).sum(), rel * float(r.norm())
        for _ in range(limit):
            q = H(p)
            a = rz / (p * q).sum()
            x, r = x + a * p, r - a * q
            if float(r.norm()) <= stop:
                break
            z = self.spectral(r, self.inv_sym)
            new = (r * z).sum()
            p, rz = z + (new / rz) * p, new
        return x

    def solve(self, u, f, g=None):
        if self.order == 6:
            u = u + (g - u).mean()
        r = self.residual(u, f, g)
        res = first = float(r.norm())
        for _ in range(100):
            if res == 0.0:
                break
            d = self.cg(self.hess(self.grad(u)), r, 1e-6)
            if self.order == 6:
                d = d - d.mean()
            t = 1.0
            while True:
                v = u + t * d
                r = self.residual(v, f, g)
                new = float(r.norm())
                if new < res or t < 1e-3:
                    break
                t *= 0.5
            if not new < res:
                break  # rounding floor: u is as good as v
            u, last, res = v, res, new
            if res > 0.5 * last and res < 1e-8 * first:
                break
        return u


def exact(case, seed):
    if case["kind"] == "batch":
        # the instances up to 128^2 (the larger ones would take minutes)
        got = {}
        for i in _batch_instances(case, seed):
            n = i["shape"][0]
            if n <= 128:
                P = _Plain(4, i["shape"], i["h"], i["p"], i["s"], i["eps"], 0.0)
                got.setdefault(n, []).append(P.solve(torch.zeros_like(i["f"]), i["f"]))
            else:
                got[n] = None
        return {str(n): None if v is None else torch.stack(v) for n, v in got.items()}
    st = _fields(case, seed)
    P = _Plain(case["order"], st["shape"], st["h"], case["p"], st["s"], case["eps"], case["lam"])
    kind = case["kind"]
    if kind == "residual":
        r = P.residual(st["u"], st["f"], st.get("g"))
        hd = st["h"] ** P.dim
        return {"r": r, "l2": float((hd * (r * r).sum()).sqrt()), "linf": float(r.abs().max())}
    if kind == "precond":
        return P.spectral(st["r"].double(), P.inv_sym)
    if kind == "solve":
        return P.solve(st["u0"], st["f"], st.get("g"))
    if kind == "grad":
        u = P.solve(st["u0"], st["f"])
        G = P.grad(u)
        lam = P.cg(P.hess(G), st["h"] ** P.dim * (u - st["target"]), 1e-14)
        ds = (P.op(u) - u) / st["s"]
        return {"u": u, "grad_f": lam, "grad_s": -(lam * ds).sum()}
    u = st["u0"]
    for _ in range(STEPS):
        if kind == "thinfilm":
            u = P.solve(u, u - st["s"] * P.div(P.grad(u)))
        else:
            u = P.solve(u, -st["s"] * 2.0 * P.lap(u), u)
    return u
