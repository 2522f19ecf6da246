"""What this library is used for, as cases that can be timed and compared.

A case is one call (or one training step, or one burst of served requests) of
the public entry points in ``paper_1901_06503_gb300``.  The sizes are those of
the workloads in ``paper_1901_06503_gb300/inputs.py``, of ``bench.py`` and of
the tests, and ragged sizes between them: the grid is set by the scanner's
resolution, so users do not get to choose a power of two.

``listed`` gives the cases, ``draw`` more of the same ranges, ``prepare`` what a
caller has in hand (inputs on the GPU and the workspace), ``run`` one pass,
``work`` the bytes and operations it cannot do without, and ``exact`` the same
outputs in 64 bits by plain torch.
"""
import math

import numpy as np
import torch

from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.autograd import forward_op

PREC = {"fp64": F.FP64, "fp32": F.FP32, "kahan": F.FP32_KAHAN}
CFL = 0.3
LAM = 1e-3

# The serving pool's requests: (n, angles, T, iterations), admitted together.
SERVE = {
    "small": ((64, 45, 0.8, 6), (64, 90, 1.1, 4), (96, 45, 0.9, 4)),
    "mixed": ((64, 90, 1.2, 6), (96, 45, 1.0, 5), (128, 90, 0.8, 4), (96, 180, 0.8, 4)),
}


def _case(name, kind, n, angles, T, prec, speed="bump", precond=0, pad=0, iters=1, every=16,
          pool=""):
    c = {"kind": kind, "n": n, "angles": angles, "T": T, "prec": prec, "speed": speed,
         "precond": precond, "pad": pad, "iters": iters, "every": every, "pool": pool}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one application of A at the smallest serving size,
        # where launches and host work count
        _case("forward-64", "forward", 64, 45, 0.8, "kahan"),
        # the plain FP64 reconstruction (32^3, 24 angles, 10 iterations)
        _case("solve-32-fp64", "solve", 32, 24, 1.0, "fp64", iters=10),
        # an odd grid and an odd number of angles: back-propagating measured data
        _case("adjoint-101", "adjoint", 101, 45, 1.0, "fp32"),
        # an even grid that is no multiple of four, random sound speed
        _case("forward-150", "forward", 150, 90, 1.0, "kahan", speed="field"),
        # the single-instance solve (128^3, 90 angles, T = 1.2), a few of its iterations
        _case("solve-128", "solve", 128, 90, 1.2, "kahan", speed="field", iters=4),
        # an iteration of the same solve in FP64, which the FP32 one is checked against
        _case("solve-128-fp64", "solve", 128, 90, 1.2, "fp64", speed="field"),
        # one step of training or descent through the differentiable operator
        # (192^3, 90 angles) with the sound speed known: data and source gradient
        _case("gradient-192", "gradient", 192, 90, 1.0, "fp32"),
        # the same with the sound speed unknown too, as it is inverted for, on a
        # coarse grid: data, source gradient and speed gradient
        _case("gradients-64", "gradients", 64, 45, 1.0, "fp32"),
        # the paper's setting in 3D: box 64^3 on a padded grid of three times
        # the width, data outside the box only, gradient regulariser
        _case("padded-64", "padded", 64, 180, 2.0, "kahan", precond=1, pad=64, iters=2),
        # plane-wise filtered backprojection of a full data set (first stage of
        # the two-step method, quick-look images)
        _case("fbp-256", "fbp", 256, 180, 1.0, "fp32"),
        # a burst of requests of different sizes through the serving loop
        _case("serve-mixed", "serve", 0, 0, 0.0, "kahan", pool="mixed"),
        # one iteration of the large preconditioned solve (384^3, 180 angles, T = 1.5)
        _case("solve-384", "solve", 384, 180, 1.5, "kahan", speed="field", precond=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind of the list over its range of sizes, odd ones among them."""
    kind = rng.choice(["forward", "adjoint", "forward", "adjoint", "solve", "solve", "gradient",
                       "gradients", "padded", "fbp", "serve"])
    T = round(rng.uniform(0.8, 1.4), 3)
    angles = _log_int(rng, 12, 180)
    speed = rng.choice(["bump", "field"])
    if kind in ("forward", "adjoint"):
        prec = rng.choice(["fp64", "fp32", "kahan"])
        n = _log_int(rng, 24, 128 if prec == "fp64" else 300)
        return _case("", kind, n, angles, T, prec, speed)
    if kind == "solve":
        prec = rng.choice(["fp64", "fp32", "kahan", "kahan"])
        n = _log_int(rng, 24, 72 if prec == "fp64" else 208)
        return _case("", kind, n, angles, T, prec, speed, rng.choice([0, 1]), 0,
                     rng.randint(1, 4))
    if kind in ("gradient", "gradients"):
        n = _log_int(rng, 32, 200 if kind == "gradient" else 72)
        return _case("", kind, n, angles, T, "fp32", speed, every=rng.choice([8, 16, 25]))
    if kind == "padded":
        n = _log_int(rng, 24, 64)
        return _case("", kind, n, angles, T, rng.choice(["fp32", "kahan"]), speed,
                     rng.choice([0, 1]), rng.randint(n // 4, n), rng.randint(1, 3))
    if kind == "fbp":
        return _case("", kind, _log_int(rng, 32, 300), angles, 1.0,
                     rng.choice(["fp32", "fp32", "fp64"]) if angles < 60 else "fp32")
    return _case("", "serve", 0, rng.randint(20, 120), T, "kahan",
                 pool=rng.choice(["small", "mixed"]))


# ------------------------------------------------------------------ inputs --
def _dtype(prec):
    return torch.float64 if prec == "fp64" else torch.float32


def _axis(n, pad=0):
    return -1.0 + (torch.arange(n + 2 * pad, dtype=torch.float64, device="cuda") - pad + 0.5) * (
        2.0 / n)


def _in_ball(rng, radius):
    while True:
        p = rng.uniform(-radius, radius, size=3)
        if p @ p <= radius * radius:
            return p


def _blobs(seed, count):
    rng = np.random.default_rng(seed)
    return [(_in_ball(rng, 0.5), rng.uniform(0.5, 1.0)) for _ in range(count)]


def _volume(n, blobs, sigma=0.08):
    """Sum of Gaussian sources (the blob phantom of the small and serving workloads)."""
    x = _axis(n)
    h = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
    for ctr, a in blobs:
        ex, ey, ez = (torch.exp(-((x - ctr[d]) ** 2) / (2 * sigma**2)) for d in range(3))
        h += a * ez[:, None, None] * ey[None, :, None] * ex[None, None, :]
    return h


def _speed(n, pad, kind, seed):
    """A Gaussian bump, or a clipped Gaussian random field; continued outwards over the padding."""
    if kind == "bump":
        ctr = _in_ball(np.random.default_rng(seed + 7), 0.3)
        x = _axis(n, pad)
        ex, ey, ez = (torch.exp(-((x - ctr[d]) ** 2) / 0.3**2) for d in range(3))
        return 1.0 + 0.2 * ez[:, None, None] * ey[None, :, None] * ex[None, None, :]
    gen = torch.Generator(device="cuda").manual_seed(seed + 7)
    w = torch.randn((n, n, n), generator=gen, dtype=torch.float64, device="cuda")
    k = 2 * math.pi * torch.fft.fftfreq(n, d=2.0 / n, dtype=torch.float64, device="cuda")
    kr = 2 * math.pi * torch.fft.rfftfreq(n, d=2.0 / n, dtype=torch.float64, device="cuda")
    s = 0.25 / math.sqrt(2.0)
    filt = torch.exp(-0.5 * s * s * (k[:, None, None] ** 2 + k[None, :, None] ** 2
                                     + kr[None, None, :] ** 2))
    f = torch.fft.irfftn(torch.fft.rfftn(w) * filt, s=(n, n, n))
    f = (f - f.mean()) / f.std()
    c = torch.clamp(1.0 + 0.15 * f, 0.8, 1.3)
    if pad:
        i = torch.clamp(torch.arange(n + 2 * pad, device="cuda") - pad, 0, n - 1)
        c = c[i][:, i][:, :, i]
    return c


def _data(n, pad, angles, T, blobs, seed, noise=0.01, sigma=0.08):
    """Projections at time T of the blobs' spherical waves in a uniform medium
    (closed form p(r, T) = [(r - T) s(r - T) + (r + T) s(r + T)] / 2r, its line
    integral tabulated over the distance from the centre) plus noise."""
    nw = n + 2 * pad
    x = _axis(n, pad)
    top = 2.0 * math.sqrt(2.0) * nw / n + 1.0
    rho = torch.linspace(0.0, top, 2048, dtype=torch.float64, device="cuda")
    line = torch.linspace(-T - 0.7, T + 0.7, 1024, dtype=torch.float64, device="cuda")
    r = torch.sqrt(rho[:, None] ** 2 + line[None, :] ** 2).clamp_min(1e-9)

    def g(u):
        return u * torch.exp(-(u**2) / (2 * sigma**2))

    table = ((g(r - T) + g(r + T)) / (2 * r)).sum(1) * float(line[1] - line[0])
    table = torch.cat([table, table[-1:]])
    out = torch.zeros((angles, nw, nw), dtype=torch.float64, device="cuda")
    th = math.pi * torch.arange(angles, dtype=torch.float64, device="cuda") / angles
    for ctr, a in blobs:
        u = x[None, :] - (ctr[0] * torch.cos(th) + ctr[1] * torch.sin(th))[:, None]
        q = torch.sqrt(u[:, None, :] ** 2 + (x - ctr[2])[None, :, None] ** 2) * (2047.0 / top)
        i = q.floor().clamp_max(2047.0)
        f = q - i
        i = i.long()
        out += a * (table[i] * (1.0 - f) + table[i + 1] * f)
    gen = torch.Generator(device="cuda").manual_seed(seed + 3)
    scale = noise * out.norm() / math.sqrt(out.numel())
    out += scale * torch.randn(out.shape, generator=gen, dtype=torch.float64, device="cuda")
    return out


def _step(case):
    """A step size below 1 / ||A||^2, as an earlier power iteration would have given it."""
    dx = 2.0 / case["n"]
    return (1.5 if case["precond"] else 0.15) / (case["angles"] * dx)


def _requests(case, seed):
    """The requests of a serving burst, as host arrays."""
    got = []
    for i, (n, angles, T, iters) in enumerate(SERVE[case["pool"]]):
        angles, T = case["angles"] or angles, case["T"] or T
        sub = _case("", "serve", n, angles, T, "kahan", iters=iters)
        blobs = _blobs(seed * 8 + i, 3)
        c = _speed(n, 0, "bump", seed * 8 + i).float().cpu().numpy()
        g = _data(n, 0, angles, T, blobs, seed * 8 + i).float().cpu().numpy()
        got.append((sub, c, g))
    return got


def _inputs(case, seed):
    """The tensors of a case, made from the seed alone."""
    n, pad, dt = case["n"], case["pad"], _dtype(case["prec"])
    kind = case["kind"]
    blobs = _blobs(seed, 8 if n > 100 else 3)
    made = {}
    if kind != "fbp":
        made["c"] = _speed(n, pad, case["speed"], seed).to(dt).contiguous()
    if kind == "forward":
        made["h"] = _volume(n, blobs).to(dt)
    if kind in ("gradient", "gradients"):
        # an early step of a training or descent loop: a blurred, weak estimate
        made["h"] = (0.5 * _volume(n, blobs, 0.12)).to(dt)
    if kind != "forward":
        made["g"] = _data(n, pad, case["angles"], case["T"], blobs, seed).to(dt)
    if kind in ("solve", "padded"):
        # a first estimate: the sources, blurred and too weak
        made["h0"] = (0.5 * _volume(n, blobs, 0.12)).to(dt)
    if kind == "padded":
        # the paper's limited data: detectors beyond the box
        m = (_axis(n, pad).abs() > 1.0).to(dt)
        made["mask"] = m.expand(case["angles"], n + 2 * pad, n + 2 * pad).contiguous()
        made["g"] *= made["mask"]
    return made


def _problem(case):
    return F.problem(case["n"], case["T"], case["angles"], PREC[case["prec"]], case["precond"],
                     CFL, case["pad"])


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"case": case, "server": F.Server(32 << 30, 8),
                "requests": [(_problem(sub), c, g, _step(sub), sub["iters"])
                             for sub, c, g in _requests(case, seed)]}
    state = _inputs(case, seed)
    prob = _problem(case)
    state.update(case=case, prob=prob)
    if "gradient" in case["kind"]:  # the differentiable operator keeps its own workspace
        state["h"].requires_grad_(True)
        state["c"].requires_grad_(case["kind"] == "gradients")
    else:
        state["ws"] = F.workspace(prob)
    return state


# --------------------------------------------------------------------- run --
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(p, c, g, LAM, step, iters)
                   for p, c, g, step, iters in state["requests"]]
        done = [server.wait(t, interval=2e-4) for t in tickets]
        return [(h, np.array([st["objective"], st["resid_norm"], st["rel_change"]], np.float32))
                for h, st in done]
    prob = state["prob"]
    if kind == "forward":
        return F.forward(prob, state["c"], state["h"], ws=state["ws"])
    if kind == "adjoint":
        return F.adjoint(prob, state["c"], state["g"], ws=state["ws"])
    if kind == "fbp":
        return F.fbp(prob, state["g"], ws=state["ws"])
    if kind in ("gradient", "gradients"):
        h, c = state["h"], state["c"]
        out = forward_op(h, c, prob, case["every"])
        loss = 0.5 * ((out - state["g"]) ** 2).sum()
        return (out.detach(), *torch.autograd.grad(loss, (h, c) if c.requires_grad else (h,)))
    if kind == "solve":
        h, _, hist = F.fb_solve(prob, state["c"], state["g"], LAM, _step(case), case["iters"],
                                h=state["h0"].clone(), ws=state["ws"])
    else:
        dx = 2.0 / case["n"]
        h, _, hist = F.fb_solve_masked(prob, state["c"], state["g"], dx * dx / _step(case),
                                       _step(case), case["iters"], mask=state["mask"],
                                       h=state["h0"].clone(), ws=state["ws"], reg=F.REG_GRAD2)
    # the history is as good as the fields it is taken from
    return h, hist if case["prec"] == "fp64" else hist.astype(np.float32)


# -------------------------------------------------------------------- work --
def _steps(case):
    cmax = {"bump": 1.2, "field": 1.3}[case["speed"]]
    return max(1, math.ceil(case["T"] * cmax * case["n"] / (2.0 * CFL)))


def work(case):
    """Inputs once and outputs once; a leapfrog step takes 10 additions and 4
    multiply-adds a point (4 additions more where the sums are compensated), a
    ray sample or its transpose 4 multiply-adds, a filtered row n / 2 a value."""
    if case["kind"] == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for n, angles, T, iters in SERVE[case["pool"]]:
            w = work(_case("", "solve", n, case["angles"] or angles, case["T"] or T, "kahan",
                           iters=iters))
            total = {k: total[k] + w[k] for k in total}
        return total
    n, nw, es = case["n"], case["n"] + 2 * case["pad"], 8 if case["prec"] == "fp64" else 4
    vol, wav, dat = n**3, nw**3, case["angles"] * nw * nw
    wave = _steps(case) * wav * (22.0 if case["prec"] == "kahan" else 18.0)
    proj = 8.0 * dat * nw
    ramp = float(dat) * nw
    kind = case["kind"]
    if kind == "forward":
        return {"bytes": es * (wav + vol + dat), "flops": wave + proj}
    if kind == "adjoint":
        return {"bytes": es * (wav + vol + dat), "flops": wave + proj}
    if kind == "fbp":
        return {"bytes": es * (wav + dat), "flops": proj + ramp}
    if kind == "gradient":
        return {"bytes": es * (3 * vol + 2 * dat), "flops": 2.0 * wave + 2 * proj}
    if kind == "gradients":
        # forward, transposed, and the product with the Laplacian of the forward field
        return {"bytes": es * (4 * vol + 2 * dat), "flops": 3.0 * wave + 2 * proj}
    prox = 12.0 * float(n) ** 4 if kind == "padded" else 0.0
    one = 2 * wave + 2 * proj + (ramp if case["precond"] else 0.0) + prox
    data = dat * (2 if kind == "padded" else 1)
    return {"bytes": es * (wav + data + 2 * vol), "flops": case["iters"] * one}


# ------------------------------------------------------------------- exact --
class _Exact:
    """The discrete operators of include/ffpat.h in 64 bits, by plain torch."""

    def __init__(self, n, pad, angles, T, c):
        self.n, self.pad, self.nw, self.angles = n, pad, n + 2 * pad, angles
        self.dx = 2.0 / n
        self.c = c.double()
        x = T * float(self.c.max()) / (CFL * self.dx)
        self.nt = max(1, math.ceil(x * (1.0 - 1e-12)))
        self.kap = (self.c * (T / self.nt / self.dx)) ** 2

    def lap(self, u):
        nw = self.nw
        v = torch.zeros((nw + 4,) * 3, dtype=torch.float64, device=u.device)
        mid = slice(2, nw + 2)
        v[mid, mid, mid] = u
        s = v[3:nw + 3, mid, mid] + v[1:nw + 1, mid, mid]
        s += v[mid, 3:nw + 3, mid]
        s += v[mid, 1:nw + 1, mid]
        s += v[mid, mid, 3:nw + 3]
        s += v[mid, mid, 1:nw + 1]
        s *= 16.0
        for lo in (0, 4):
            s -= v[lo:lo + nw, mid, mid]
            s -= v[mid, lo:lo + nw, mid]
            s -= v[mid, mid, lo:lo + nw]
        s.add_(u, alpha=-90.0)
        return s.mul_(1.0 / 12.0)

    def wave(self, h, kap=None, keep=None):
        """T_Nt of the leapfrog recurrence; kap applied outside the Laplacian."""
        kap = self.kap if kap is None else kap
        if keep is not None:
            keep.append(h)
        a, b = h, h + 0.5 * kap * self.lap(h)
        for _ in range(self.nt - 1):
            if keep is not None:
                keep.append(b)
            s = self.lap(b).mul_(kap)
            s += 2.0 * b
            s -= a
            a, b = b, s
        return b

    def wave_t(self, q):
        return self.wave(self.kap * q) / self.kap

    def embed(self, h):
        p = self.pad
        if not p:
            return h
        out = torch.zeros((self.nw,) * 3, dtype=torch.float64, device=h.device)
        out[p:-p, p:-p, p:-p] = h
        return out

    def restrict(self, u):
        p = self.pad
        return u[p:-p, p:-p, p:-p] if p else u

    def _corners(self, j):
        """Plane indices (of a plane with a zero border) and weights of the samples of angle j."""
        nw, dx = self.nw, self.dx
        L, ns = nw / self.n, 2 * math.ceil(nw / math.sqrt(2.0))
        th = math.pi * j / self.angles
        cs, sn = math.cos(th), math.sin(th)
        xi = -L + (torch.arange(nw, dtype=torch.float64, device="cuda") + 0.5) * dx
        s = (torch.arange(ns, dtype=torch.float64, device="cuda") + 0.5 - ns // 2) * dx
        gx = (xi[:, None] * cs - s[None, :] * sn + L) / dx - 0.5
        gy = (xi[:, None] * sn + s[None, :] * cs + L) / dx - 0.5
        i, k = gx.floor(), gy.floor()
        fx, fy = gx - i, gy - k
        at, w = [], []
        for dy in (0, 1):
            for dxi in (0, 1):
                ii = (i + dxi).clamp(-1, nw).long() + 1
                kk = (k + dy).clamp(-1, nw).long() + 1
                at.append(kk * (nw + 2) + ii)
                w.append((fx if dxi else 1.0 - fx) * (fy if dy else 1.0 - fy))
        return torch.cat(at, 1), torch.cat(w, 1)

    def project(self, u):
        nw = self.nw
        t = torch.zeros((nw + 2, nw + 2, nw), dtype=torch.float64, device=u.device)
        t[1:-1, 1:-1] = u.permute(1, 2, 0)
        t = t.view(-1, nw)
        out = torch.empty((self.angles, nw, nw), dtype=torch.float64, device=u.device)
        for j in range(self.angles):
            at, w = self._corners(j)
            out[j] = torch.nn.functional.embedding_bag(at, t, per_sample_weights=w,
                                                       mode="sum").t()
        return out * self.dx

    def project_t(self, g):
        nw = self.nw
        t = torch.zeros(((nw + 2) ** 2, nw), dtype=torch.float64, device=g.device)
        for j in range(self.angles):
            at, w = self._corners(j)
            rows = g[j].t().contiguous()
            part = max(1, (1 << 28) // (at.shape[1] * nw))  # bounds the temporary
            for k in range(0, nw, part):
                t.index_add_(0, at[k:k + part].reshape(-1),
                             (w[k:k + part, :, None] * rows[k:k + part, None, :]).view(-1, nw))
        u = t.view(nw + 2, nw + 2, nw)[1:-1, 1:-1].permute(2, 0, 1)
        return u.contiguous() * self.dx

    def ramp(self, r):
        nw = self.nw
        d = torch.arange(nw, dtype=torch.float64, device=r.device)
        t = torch.where(d % 2 == 1, -1.0 / (2 * math.pi**2 * d.clamp_min(1) ** 2 * self.dx),
                        torch.zeros_like(d))
        t[0] = 1.0 / (8.0 * self.dx)
        i = torch.arange(nw, device=r.device)
        return r @ t[(i[:, None] - i[None, :]).abs()]

    def grad_energy(self, h):
        return 0.5 * sum(float((h.diff(dim=d) ** 2).sum()) for d in range(3)) / self.dx**2

    def prox_grad(self, f, a):
        n = self.n
        i = torch.arange(n, dtype=torch.float64, device=f.device)
        C = torch.cos(math.pi * i[:, None] * (2 * i[None, :] + 1) / (2 * n)) * math.sqrt(2.0 / n)
        C[0] /= math.sqrt(2.0)
        mu = 4.0 * torch.sin(math.pi * i / (2 * n)) ** 2
        F3 = torch.einsum("ai,bj,ck,ijk->abc", C, C, C, f)
        F3 /= 1.0 + a * (mu[:, None, None] + mu[None, :, None] + mu[None, None, :])
        return torch.einsum("ai,bj,ck,abc->ijk", C, C, C, F3)

    def solve(self, g, h, lam, step, iters, precond, mask=None, grad2=False):
        g, h, hist = g.double(), h.double(), []
        for _ in range(iters):
            r = self.project(self.wave(self.embed(h))) - g
            if mask is not None:
                r = r * mask
            lr = self.ramp(r) if precond else r
            if precond and mask is not None:
                lr = lr * mask
            grad = self.restrict(self.wave_t(self.project_t(lr)))
            f = h - step * grad
            if grad2:
                reg, new = self.grad_energy(h), self.prox_grad(f, step * lam / self.dx**2)
            else:
                reg, new = float(h.abs().sum()), torch.clamp(f - step * lam, min=0.0)
            hist.append([0.5 * float((lr * r).sum()) + lam * reg, float(r.norm()),
                         float((new - h).norm()) / max(float(h.norm()), 1e-300),
                         float(new.norm())])
            h = new
        return h, np.array(hist)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        got = []
        for sub, c, g in _requests(case, seed):
            e = _Exact(sub["n"], 0, sub["angles"], sub["T"], torch.as_tensor(c, device="cuda"))
            g = torch.as_tensor(g, device="cuda")
            h, hist = e.solve(g, torch.zeros_like(e.c), LAM, _step(sub), sub["iters"], 0)
            got.append((h, hist[-1][:3]))
        return got
    made = _inputs(case, seed)
    n, pad, angles = case["n"], case["pad"], case["angles"]
    if kind == "fbp":
        e = _Exact(n, 0, angles, case["T"], torch.ones((1, 1, 1), device="cuda"))
        return e.project_t(e.ramp(made["g"].double())) * (2.0 * math.pi / (angles * e.dx))
    e = _Exact(n, pad, angles, case["T"], made["c"])
    if kind == "forward":
        return e.project(e.wave(e.embed(made["h"].double())))
    if kind == "adjoint":
        return e.restrict(e.wave_t(e.project_t(made["g"].double())))
    if kind == "gradient":
        out = e.project(e.wave(made["h"].double()))
        return out, e.wave_t(e.project_t(out - made["g"].double()))
    if kind == "gradients":
        kept = []
        out = e.project(e.wave(made["h"].double(), keep=kept))
        # lam^n = 2 lam^{n+1} - lam^{n+2} + L(kap lam^{n+1}), and the derivative
        # in kap gathers lam^{n+1} L(p^n) (half of it at the start step)
        b = e.project_t(out - made["g"].double())
        a = torch.zeros_like(b)
        gk = torch.zeros_like(b)
        for s in range(e.nt - 1, 0, -1):
            gk += b * e.lap(kept[s])
            a, b = b, 2.0 * b - a + e.lap(e.kap * b)
        gk += 0.5 * b * e.lap(kept[0])
        gh = b - a + 0.5 * e.lap(e.kap * b)
        return out, gh, gk * 2.0 * e.kap / e.c
    lam, step = LAM, _step(case)
    if kind == "padded":
        lam = e.dx**2 / step
    return e.solve(made["g"], made["h0"], lam, step, case["iters"], case["precond"],
                   made.get("mask"), kind == "padded")
