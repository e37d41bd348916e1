"""Workloads of the ETD membrane library, measured and checked: the calls that a program makes
through `Plan` and `Batch`, over the sizes, models, schemes and precisions the library takes.

Kinds of case:
  coupled  `Plan.step` of the phi-u system (Algorithm 1), 3D
  fixed    `Plan.step` of the protein density on a frozen membrane (Sec. 3 split), 2D and 3D
  sqrtg    `Plan.step` of the Sec. 2.2 scheme on a frozen membrane (Krylov), 2D and 3D
  batch    `Batch.step` of independent frozen-membrane runs on uneven grids
  energy   `Plan.energy`, the diagnostics of a state
  fft      `Plan.fft_forward` and `Plan.fft_inverse`
A stepping pass starts from the state it is handed (copied into the buffers that the plan
advances), so that every pass does the same work and long sequences of passes stay in the part
of a run where the model is stable.
"""
import math

import torch

from paper_2606_04347_gb300 import Batch, Plan
from paper_2606_04347_gb300 import workloads as wl

LENGTHS = (8, 16, 32, 64, 96, 128, 256)


def _case(name, kind, n, prec, scheme=2, steps=1, eps=0.05, tau=1e-3, gamma=100.0, B2=2000.0, shape="circle", runs=0):
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], prec=prec, scheme=scheme, steps=steps, eps=eps, tau=tau, gamma=gamma,
             B2=B2, shape=shape, runs=runs)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one step of the smallest practical grid: a program that looks at every step (launches, latency)
        _case("fixed_2d_64_etd1_fp32", "fixed", (64, 64, 1), 32, scheme=1, eps=0.1),
        # the 2D frozen-membrane run: circle, ETD1, double precision
        _case("fixed_2d_128_etd1_fp64", "fixed", (128, 128, 1), 64, scheme=1, steps=10),
        # uneven extents, one of them 96, as sweeps over boxes and resolutions have them
        _case("fixed_96x128x64_fp32", "fixed", (96, 128, 64), 32, steps=4, tau=2e-3, gamma=60.0, B2=4000.0),
        # the 3D frozen sphere, ETDRK2, double precision
        _case("fixed_128_fp64", "fixed", (128, 128, 128), 64, steps=4, tau=1.25e-3),
        # the paper's 2D rate-study setting with the Sec. 2.2 scheme
        _case("sqrtg_2d_256_fp64", "sqrtg", (256, 256, 1), 64, steps=4, eps=10.0, tau=1e-4),
        # coupled runs from a trial resolution to the full one
        _case("coupled_64_fp32", "coupled", (64, 64, 64), 32, steps=4, eps=0.18, tau=1e-4),
        _case("coupled_128_etd1_fp32", "coupled", (128, 128, 128), 32, scheme=1, steps=6, eps=0.18, tau=1e-4),
        _case("coupled_256_fp32", "coupled", (256, 256, 256), 32, steps=8, eps=0.18, tau=1e-4),
        # the double-precision coupled form, used to check the mixed one
        _case("coupled_128_fp64", "coupled", (128, 128, 128), 64, steps=3, eps=0.18, tau=1e-4),
        # a parameter sweep: eight runs on 64^3, 96^3 and 128^3 advanced together
        _case("batch_8_fp32", "batch", (128, 128, 128), 32, steps=12, runs=8),
        # diagnostics of a full-resolution state, taken between stretches of a run
        _case("energy_256_fp32", "energy", (256, 256, 256), 32, eps=0.18),
        # transforms of a full-resolution field, to and from the half spectrum
        _case("fft_256_fp32", "fft", (256, 256, 256), 32),
    ]


def draw(rng):
    kind = rng.choice(("coupled", "coupled", "fixed2d", "fixed3d", "sqrtg", "batch", "energy", "fft"))
    prec, scheme = rng.choice((32, 32, 64)), rng.choice((1, 2, 2))
    if kind == "coupled":
        big = 2 ** rng.randint(15, 24 if prec == 32 else 21)
        while True:
            n = [rng.choice((32, 64, 128, 256)) for _ in range(3)]
            if prec == 64:
                n = [rng.choice((v, 96) if v in (64, 128) else (v,)) for v in n]
            if big / 2 <= n[0] * n[1] * n[2] <= big:
                break
        return _case("", "coupled", n, prec, scheme, rng.randint(1, 6), 0.18, rng.choice((5e-5, 1e-4)))
    if kind == "fixed2d":
        n = [rng.choice((32, 64, 96, 128, 256)) for _ in range(2)]
        return _case("", "fixed", (*n, 1), prec, scheme, rng.randint(1, 12), rng.uniform(0.6, 1.2) * 2 * math.pi / min(n), 1e-3)
    if kind in ("fixed3d", "energy"):
        n = [rng.choice((32, 64, 96, 128)) for _ in range(3)]
        eps = rng.uniform(0.6, 1.0) * 2 * math.pi / min(n)
        return _case("", kind[:5] if kind == "fixed3d" else kind, n, prec, scheme, rng.randint(1, 4), eps, rng.choice((1e-3, 2e-3)),
                     rng.uniform(10.0, 200.0), 4000.0 * rng.choice((1, 2, 4)))
    if kind == "sqrtg":
        if rng.random() < 0.7:
            n = rng.choice((64, 96, 128, 256))
            return _case("", "sqrtg", (n, n, 1), prec, scheme, rng.randint(1, 4), rng.uniform(5.0, 15.0), 1e-4,
                         shape=rng.choice(("circle", "ellipse", "wavy")))
        n = [rng.choice((32, 64)) for _ in range(3)]
        return _case("", "sqrtg", n, prec, scheme, 1, rng.uniform(5.0, 10.0), 1e-4)
    if kind == "batch":
        return _case("", "batch", (128, 128, 128), 32, steps=rng.randint(8, 14), runs=rng.randint(2, 8))
    two = rng.random() < 0.3
    n = [rng.choice(LENGTHS) for _ in range(3)]
    if prec == 64:
        n = [min(v, 128) for v in n]
    return _case("", "fft", (n[0], n[1], 1 if two else n[2]), prec)


# ---- inputs -----------------------------------------------------------------------------


def _params(c):
    dim = 2 if c["nz"] == 1 else 3
    p = wl.ModelParams(dim=dim, n=(c["nx"], c["ny"], c["nz"]), scheme=c["scheme"], precision=0 if c["prec"] == 64 else 1,
                       tau=c["tau"], cg_rtol=1e-12 if c["prec"] == 64 else 1e-6)
    if c["kind"] == "sqrtg":  # [-1, 1]^d, eps_phi = 10 h (3D: 5 h), eps_u = eps h of the coarsest axis
        h = 2.0 / min(p.n[:dim])
        return p.replace(model=2, half_len=(1.0,) * 3, eps_phi=(10 if dim == 2 else 5) * h, eps_u=c["eps"] * h, gamma=100.0, B2=2000.0, B1=1.0,
                         M=600.0 if c["scheme"] == 1 else 200.0, ubar=0.3)
    eps_phi, eps_u = wl.eps_from_cfg(c["eps"])
    p = p.replace(half_len=(math.pi,) * 3, eps_phi=eps_phi, eps_u=eps_u)
    if c["kind"] == "coupled":
        if c["prec"] == 32:
            p = p.replace(cg_rtol=1e-4, cg_rtol_pred=1e-4)
        return p.replace(model=1, mu=500.0)
    return p.replace(model=0, gamma=c["gamma"], M=600.0 if c["scheme"] == 1 else 200.0, ubar=0.5, B1=1.0, B2=c["B2"])


def _axes(p):
    """Coordinates along (z,) y, x, each shaped to broadcast over the field."""
    out = []
    for k, d in enumerate(reversed(range(p.dim))):
        x = -p.half_len[d] + torch.arange(p.n[d], dtype=torch.float64, device="cuda") * (2 * p.half_len[d] / p.n[d])
        out.append(x.reshape([-1 if j == k else 1 for j in range(p.dim)]))
    return out


def _fields(c, p, seed):
    """phi and u in the plan's precision: a tanh membrane of seeded size, and a protein density
    of seeded noise (frozen membranes, as their runs start) or of seeded waves (coupled runs, as
    they look once the first steps have smoothed the noise)."""
    gen = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)
    rnd = torch.rand(64, generator=gen, device="cuda", dtype=torch.float64).tolist()
    ax = _axes(p)
    X = p.half_len[0]
    if c["kind"] == "coupled" or (c["kind"] == "energy" and c["eps"] == 0.18):
        a = [1.2 + 0.06 * (rnd[0] - 0.5), 0.9 + 0.06 * (rnd[1] - 0.5), 0.9 + 0.06 * (rnd[2] - 0.5)]
        r0, r = a[0], torch.sqrt(sum((a[0] / a[2 - k] * x) ** 2 for k, x in enumerate(ax)))
    elif c["kind"] == "sqrtg":
        y, x = ax[-2:]
        r0 = 0.4 * (1 + 0.1 * (rnd[0] - 0.5))
        if c["shape"] == "wavy":
            r0 = r0 * (1 + 0.1 * torch.sin(7 * torch.atan2(y, x)))
        w = math.sqrt(3.0) if c["shape"] == "ellipse" else 1.0
        r = torch.sqrt(x * x + w * y * y + (ax[0] ** 2 if p.dim == 3 else 0.0))
    else:
        r0, r = (0.6 if p.dim == 2 else 0.5) * math.pi * (1 + 0.04 * (rnd[0] - 0.5)), torch.sqrt(sum(x * x for x in ax))
    phi = (0.5 + 0.5 * torch.tanh(3 * (r0 - r) / p.eps_phi)).expand(p.shape).contiguous()
    if c["kind"] in ("coupled", "sqrtg") or (c["kind"] == "energy" and c["eps"] == 0.18):
        s = torch.zeros(p.shape, dtype=torch.float64, device="cuda")
        for k in range(5):  # plane waves, up to five periods a side
            arg = 2 * math.pi * rnd[8 + 8 * k]
            for j, x in enumerate(ax):
                arg = arg + math.pi / X * round(10 * rnd[9 + 8 * k + j] - 5) * x
            s += torch.sin(arg)
        u = 0.5 + 0.08 * s
        if c["kind"] != "sqrtg":  # off the recovery set the state holds G u
            G = 18 * (phi * phi - phi) ** 2
            u = torch.where(G > p.recover_delta, u, G * u)
    elif p.dim == 2:
        u = 0.5 * (1 + 0.2 * (torch.rand(p.shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5))
    else:
        u = 0.5 * (1 + (0.1 * torch.randn(p.shape, generator=gen, device="cuda", dtype=torch.float64)).clamp(-1, 1))
    t = torch.float64 if c["prec"] == 64 else torch.float32
    return phi.to(t), u.to(t)


def _sweep(c, seed):
    """The runs of a batch: grids, widths, strengths and steps as a parameter sweep mixes them."""
    gen = torch.Generator().manual_seed(7919 * c["runs"] + c["steps"])  # which runs: the same for every seed
    pick = torch.rand(c["runs"], 5, generator=gen).tolist()
    out = []
    for i, r in enumerate(pick):
        n = (64, 96, 128)[(i + int(3 * r[0])) % 3]
        q = dict(c, kind="fixed", nx=n, ny=n, nz=n, eps=0.05 + 0.03 * r[1], gamma=10 + 190 * r[2], B2=4000.0 * (1, 2, 4)[int(3 * r[3])],
                 tau=(1e-3, 2e-3)[int(2 * r[4])])
        p = _params(q)
        out.append((q, p, *_fields(q, p, 101 * int(seed) + i)))
    return out


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        runs = _sweep(c, seed)
        phis, us = [r[2] for r in runs], [r[3] for r in runs]
        return dict(c=c, batch=Batch([r[1] for r in runs]), phis=phis, start=us, us=[u.clone() for u in us])
    if c["kind"] == "fft":
        p = _params(c)
        t = torch.float64 if c["prec"] == 64 else torch.float32
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        f = torch.rand(p.shape, generator=gen, device="cuda", dtype=t)
        half = torch.zeros(*p.shape[:-1], p.n[0] // 2 + 1, dtype=torch.complex128 if c["prec"] == 64 else torch.complex64, device="cuda")
        return dict(c=c, plan=Plan(p), f=f, half=half, back=torch.empty_like(f))
    p = _params(c)
    phi, u = _fields(c, p, seed)
    plan = Plan(p)
    if c["kind"] in ("fixed", "sqrtg"):  # the membrane is handed over once, before the steps
        plan.step(phi, u, 0)
    return dict(c=c, plan=plan, phi0=phi, u0=u, phi=phi.clone(), u=u.clone())


def run(s):
    c = s["c"]
    if c["kind"] == "batch":
        for u, u0 in zip(s["us"], s["start"]):
            u.copy_(u0)
        s["batch"].step(s["phis"], s["us"], c["steps"])
        return s["us"]
    if c["kind"] == "fft":
        s["plan"].fft_forward(s["f"], s["half"])
        s["plan"].fft_inverse(s["half"], s["back"])
        return s["half"], s["back"]
    if c["kind"] == "energy":
        d = s["plan"].energy(s["phi0"], s["u0"])
        return {k: d[k] for k in ("energy", "mass", "max_bound", "umin", "umax", "volume", "band_size")}
    s["u"].copy_(s["u0"])
    if c["kind"] == "coupled":
        s["phi"].copy_(s["phi0"])
        s["plan"].step(s["phi"], s["u"], c["steps"])
        return s["phi"], s["u"]
    s["plan"].step(None, s["u"], c["steps"])
    return s["u"]


def work(case):
    """Each step reads and writes its state once (a frozen membrane is read only), and takes its
    real transforms at 2.5 N log2 N operations each; band solves are not counted."""
    c, size = case, 8 if case["prec"] == 64 else 4
    if c["kind"] == "batch":
        per = [work(q) for q, *_ in _sweep_sizes(c)]
        return {k: sum(w[k] for w in per) for k in ("bytes", "flops")}
    N = c["nx"] * c["ny"] * c["nz"]
    one = 2.5 * N * math.log2(N)
    if c["kind"] == "fft":
        return {"bytes": (2 * N + 2 * (c["nx"] // 2 + 1) * 2 * c["ny"] * c["nz"]) * size, "flops": 2 * one}
    if c["kind"] == "energy":
        return {"bytes": 2 * N * size, "flops": 30 * N}
    if c["kind"] == "sqrtg":
        return {"bytes": 3 * N * size * c["steps"], "flops": 30 * N * c["steps"]}
    rk2 = c["scheme"] == 2
    k, fields = ((19, 4) if rk2 else (10, 4)) if c["kind"] == "coupled" else ((5, 3) if rk2 else (3, 3))
    return {"bytes": fields * N * size * c["steps"], "flops": k * one * c["steps"]}


def _sweep_sizes(c):
    gen = torch.Generator().manual_seed(7919 * c["runs"] + c["steps"])
    for i, r in enumerate(torch.rand(c["runs"], 5, generator=gen).tolist()):
        n = (64, 96, 128)[(i + int(3 * r[0])) % 3]
        yield (dict(c, kind="fixed", nx=n, ny=n, nz=n),)


# ---- the same results in plain 64-bit torch -----------------------------------------------


def _dW(s):
    return 36 * s * (s - 1) * (2 * s - 1)


def _g(f):
    return 18 * (f * f - f) ** 2


def _f(u):
    return 3 * u * u - 2 * u ** 3


def _phis(z):
    """phi_0, phi_1, phi_2: series below 1, closed forms above."""
    s = z.clamp(max=1.0)
    p1, p2 = torch.zeros_like(z), torch.zeros_like(z)
    for k in reversed(range(26)):
        p1, p2 = p1 + (-s) ** k / float(math.factorial(k + 1)), p2 + (-s) ** k / float(math.factorial(k + 2))
    big = z.clamp(min=1.0)
    em = torch.expm1(-big)
    return torch.exp(-z), torch.where(z < 1, p1, -em / big), torch.where(z < 1, p2, (em + big) / big ** 2)


class _Exact:
    """The method on one grid (fields in double precision, x along the last axis)."""

    def __init__(self, p):
        self.p, self.dims = p, list(range(p.dim))
        self.h = p.h[:p.dim]
        self.w = None
        ks, m, self.deriv = math.pi / p.half_len[0], 0, []
        for d in range(p.dim):
            n = p.n[d]
            i = torch.arange(n // 2 + 1 if d == 0 else n, device="cuda")
            fold = torch.where(i <= n // 2, i, n - i)
            sign = torch.where(i < n // 2, i, torch.where(i == n // 2, 0, i - n))
            shape = [-1 if j == p.dim - 1 - d else 1 for j in range(p.dim)]
            m = m + (fold * fold).reshape(shape)
            self.deriv.append(1j * ks * sign.to(torch.float64).reshape(shape))
        self.lam = -ks * ks * m.to(torch.float64)
        lu = p.B2 - p.eps_u * p.B1 * self.lam
        self.cu = [a * b for a, b in zip(_phis(p.tau * lu), (1, p.tau, p.tau))]
        if p.model == 1:
            e2, lam = p.eps_phi ** 2, self.lam
            lphi = (p.kappa / p.mu * lam * lam - (p.kappa * (p.A1 + p.A2) + p.lambda_surf * e2) / (p.mu * e2) * lam
                    + (p.kappa * p.A1 * p.A2 + p.lambda_surf * p.A1 * e2) / (p.mu * e2 * e2))
            self.cphi = [a * b for a, b in zip(_phis(p.tau * lphi), (1, p.tau, p.tau))]

    def fft(self, v):
        return torch.fft.rfftn(v, dim=self.dims)

    def ifft(self, v):
        return torch.fft.irfftn(v, s=self.p.shape, dim=self.dims)

    def sh(self, v, d, k):
        return torch.roll(v, -k, self.p.dim - 1 - d)

    def surf(self, u, g):
        out = 0
        for d, h in enumerate(self.h):
            up, um, gp, gm = self.sh(u, d, 1), self.sh(u, d, -1), self.sh(g, d, 1), self.sh(g, d, -1)
            out = out + (0.5 * (gp + g) * (up - u) - 0.5 * (g + gm) * (u - um)) / (h * h)
        return out

    def lap(self, v):
        return sum((self.sh(v, d, 1) - 2 * v + self.sh(v, d, -1)) / (h * h) for d, h in enumerate(self.h))

    def inner(self, a):
        return math.prod(self.h) * float(a.sum())

    def set_band(self, phi, g):
        """The band's nodes, face couplings and neighbours (zero flux across its edge)."""
        p = self.p
        mask = (2 * phi - 1).abs() < p.band_mask_hi
        self.mask, self.idx = mask, mask.reshape(-1).nonzero().reshape(-1)
        M = self.idx.numel()
        num = torch.zeros(mask.numel(), dtype=torch.int64, device="cuda")
        num[self.idx] = torch.arange(M, device="cuda")
        num = num.reshape(mask.shape)
        own = torch.arange(M, device="cuda")
        self.nb, self.cf = [], []
        for d, h in enumerate(self.h):
            for k in (1, -1):
                on = self.sh(mask, d, k).reshape(-1)[self.idx]
                self.nb.append(torch.where(on, self.sh(num, d, k).reshape(-1)[self.idx], own))
                self.cf.append(torch.where(on, 0.5 * (g + self.sh(g, d, k)).reshape(-1)[self.idx] / (h * h), 0.0))
        self.nb, self.cf = torch.stack(self.nb), torch.stack(self.cf)
        self.diag = self.cf.sum(0)

    def neg_lap(self, x):
        return self.diag * x - (self.cf * x[self.nb]).sum(0)

    def solve(self, f, rtol=1e-13):
        """w = (-Delta_S)^{-1}(f - mean) on the band, zero mean (the band is connected)."""
        b = f.reshape(-1)[self.idx]
        b = b - b.mean()
        x = torch.zeros_like(b) if self.w is None else self.w.reshape(-1)[self.idx].clone()
        r = b - self.neg_lap(x)
        z = r / self.diag
        q, rz, bb = z, (r * z).sum(), (b * b).sum()
        for k in range(6000):
            Aq = self.neg_lap(q)
            a = rz / (q * Aq).sum()
            x, r = x + a * q, r - a * Aq
            if k % 16 == 15 and float((r * r).sum()) <= rtol * rtol * float(bb):
                break
            z = r / self.diag
            rz, old = (r * z).sum(), rz
            q = z + (rz / old) * q
        self.w = torch.zeros(f.numel(), dtype=f.dtype, device="cuda")
        self.w[self.idx] = x - x.mean()
        self.w = self.w.reshape(f.shape)
        return self.w

    def R1(self, phi, u):
        p, e = self.p, self.p.eps_phi
        P = self.fft(phi)
        lap, gn = self.ifft(self.lam * P), torch.sqrt(sum(self.ifft(s * P) ** 2 for s in self.deriv))
        Wp, Wpp = _dW(phi), 36 * (6 * phi * phi - 6 * phi + 1)
        Wm, g = Wp - p.A1 * phi, _g(phi)
        r = (p.kappa / (p.mu * e * e) * (self.ifft(self.lam * self.fft(Wm)) + (Wpp - p.A2) * (lap - p.A1 * phi / (e * e)))
             - (p.kappa * Wpp / (p.mu * e ** 4) + p.lambda_surf / (p.mu * e * e)) * Wm)
        line = (p.lambda_line / p.mu) * (p.eps_u * self.surf(u, g) - g * _dW(u) / p.eps_u) * gn
        r = r + torch.where((2 * phi - 1).abs() < p.band_mask_hi, line, 0.0)
        r = r - (p.M_area / p.mu) * (self.inner(phi) - self.A0) * gn
        return r + (p.alpha / p.mu) * (u + p.u0) * gn * (e * lap - Wp / e)

    def R2(self, u, g, phin=None, phio=None):
        p, gu = self.p, g * u
        r = p.eps_u * (self.surf(u, g) - p.B1 * self.lap(gu)) + p.B2 * gu - g * _dW(u) / p.eps_u
        if phin is None:
            fp = 6 * u * (1 - u)
            r = r - p.gamma * g * fp * self.solve(g * _f(u)) - p.M * g * fp * self.inner(g * (_f(u) - p.ubar))
        else:
            r = r - p.gamma * g * self.solve(g * (u - p.ubar)) - p.M * g * self.inner(g * (u - p.ubar))
            gr = [(self.sh(phin, d, 1) - self.sh(phin, d, -1)) / (2 * h) for d, h in enumerate(self.h)]
            s = -gu * (phin - phio) / p.tau / (sum(x * x for x in gr) + 1e-12)
            for d, h in enumerate(self.h):
                r = r - (self.sh(s * gr[d], d, 1) - self.sh(s * gr[d], d, -1)) / (2 * h)
        return torch.where(self.mask, r, 0.0)

    def recover(self, GU, G):
        return torch.where(G > self.p.recover_delta, GU / torch.where(G > self.p.recover_delta, G, 1.0), GU)

    def u_stage(self, u, G, phin=None, phio=None):
        b0, b1, b2 = self.cu
        Rn = self.fft(self.R2(u, G, phin, phio))
        GU = b0 * self.fft(G * u) + b1 * Rn
        if self.p.scheme == 2:
            ut = self.recover(self.ifft(GU), G)
            GU = GU + b2 * (self.fft(self.R2(ut, G, phin, phio)) - Rn)
        return self.recover(self.ifft(GU), G)

    def coupled(self, phi, u, steps):
        self.A0 = self.inner(phi)
        a0, a1, a2 = self.cphi
        for _ in range(steps):
            Rn = self.fft(self.R1(phi, u))
            P = a0 * self.fft(phi) + a1 * Rn
            if self.p.scheme == 2:
                P = P + a2 * (self.fft(self.R1(self.ifft(P), u)) - Rn)
            new = self.ifft(P)
            G = _g(new)
            if self.w is not None:
                self.w = torch.where((2 * new - 1).abs() < self.p.band_mask_hi, self.w, 0.0)
            self.set_band(new, G)
            phi, u = new, self.u_stage(u, G, new, phi)
        return phi, u

    def fixed(self, phi, u, steps):
        G = _g(phi)
        self.set_band(phi, G)
        for _ in range(steps):
            u = self.u_stage(u, G)
        return u

    def krylov(self, b, j, m=64):
        """tau phi_j(tau L) b by the Lanczos process with full reorthogonalisation."""
        nrm = b.norm()
        V, T = [b / nrm], torch.zeros(m, m, dtype=torch.float64)
        for k in range(m):
            w = self.L(V[k])
            Q = torch.stack(V)
            T[k, k] = float((w * V[k]).sum())
            for _ in range(2):
                w = w - Q.t() @ (Q @ w)
            if k + 1 < m:
                T[k, k + 1] = T[k + 1, k] = float(w.norm())
                V.append(w / w.norm())
        lam, S = torch.linalg.eigh(T)
        y = S @ (_phis(self.p.tau * lam.clamp(min=0))[j] * S[0])
        return self.p.tau * nrm * (torch.stack(V).t() @ y.cuda())

    def L(self, x):
        return self.p.B2 * x + self.p.eps_u / self.sg * self.neg_lap(x / self.sg)

    def sqrtg(self, phi, u, steps):
        p, G = self.p, _g(phi)
        self.set_band(phi, G)
        self.sg = torch.sqrt(G.reshape(-1)[self.idx])

        def R(v):
            w = self.solve(G * _f(v)).reshape(-1)[self.idx]
            mass = self.inner(G * (_f(v) - p.ubar))
            x = v.reshape(-1)[self.idx]
            fp = 6 * x * (1 - x)
            return self.sg * (p.B2 * x - _dW(x) / p.eps_u - p.gamma * fp * w - p.M * mass * fp)

        def put(v, V):
            out = v.reshape(-1).clone()
            out[self.idx] = V / self.sg
            return out.reshape(v.shape)

        for _ in range(steps):
            V, R0 = self.sg * u.reshape(-1)[self.idx], R(u)
            V = V + self.krylov(R0 - self.L(V), 1)
            ut = put(u, V)
            u = put(u, V + self.krylov(R(ut) - R0, 2)) if p.scheme == 2 else ut
        return u

    def energy(self, phi, u):
        p, g = self.p, _g(phi)
        self.set_band(phi, g)
        grad = sum(0.5 * (g + self.sh(g, d, 1)) * (self.sh(u, d, 1) - u) ** 2 / (h * h) for d, h in enumerate(self.h))
        mass, on = self.inner(g * (_f(u) - p.ubar)), u[g > p.recover_delta]
        e = (0.5 * p.eps_u * self.inner(grad) + self.inner(g * _g(u)) / p.eps_u
             + 0.5 * p.gamma * self.inner(self.solve(g * _f(u)) * g * _f(u)) + 0.5 * p.M * mass * mass)
        return {"energy": e, "mass": mass, "max_bound": float((2 * on - 1).abs().max()), "umin": float(on.min()),
                "umax": float(on.max()), "volume": self.inner(phi), "band_size": self.idx.numel()}


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        return [_Exact(p).fixed(phi.double(), u.double(), c["steps"]) for _, p, phi, u in _sweep(c, seed)]
    p = _params(c)
    if c["kind"] == "fft":
        t = torch.float64 if c["prec"] == 64 else torch.float32
        f = torch.rand(p.shape, generator=torch.Generator(device="cuda").manual_seed(int(seed)), device="cuda", dtype=t).double()
        return torch.fft.rfftn(f), f
    phi, u = (v.double() for v in _fields(c, p, seed))
    if c["kind"] == "energy":
        return _Exact(p).energy(phi, u)
    return getattr(_Exact(p), c["kind"])(phi, u, *([c["steps"]]))
