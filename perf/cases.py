"""The workloads that this framework's speed is measured on.

A pass takes a run (or a batch, or a stream of requests) from the fields it
starts from through a few time steps, each solved to the default 1e-10, and
hands the new state back, all through the public calls.  The sizes and
parameters are those of the repository's own configurations: the 64^2 and
512^2 spinodal runs, the gamma study, the 128^3 bubbles, the batched runs of
64^2 ... 1024^2 and the serving stream of 128^2 ... 2048^2 and 64^3 ... 256^3.

Fields: "noise" is the start of a run (rough spinodal noise), "domains" what
most of a run's steps see (separated phases with tanh interfaces, slightly
moved from one level to the next), "bubbles" the 3D workload's tanh spheres.
"""
import math
import random

import numpy as np
import torch

from paper_1611_02967_gb300 import chhs


def listed():
    return [
        # a small run's first steps: launches and latency
        _single("spinodal64_f64", (64, 64), 0, 5, "noise", 0.05, 0.05, 1.0, 0.01),
        # the gamma study's loop: a step, then energies, mass and dissipation, in double precision
        _single("study512_f64", (512, 512), 0, 2, "noise", 0.0125, 0.03, 2.0, 0.01, diagnostics=True),
        # the 512^2 run in both forms, phases separated
        _single("spinodal512_f64", (512, 512), 0, 3, "domains", 0.025, 0.05, 1.0, 0.005),
        _single("spinodal512_mixed", (512, 512), 1, 4, "domains", 0.025, 0.05, 1.0, 0.005),
        # a rectangle that is no power of two (coarsens to 5 x 3)
        _single("ragged640x384_mixed", (384, 640), 1, 4, "domains", 0.025, 0.04, 2.0, 0.005),
        # the largest 2D run of the serving stream
        _single("served2048_mixed", (2048, 2048), 1, 2, "noise", 0.025, 0.06, 1.5, 0.005),
        # a box of the serving stream's smaller 3D sizes, sides no powers of two (coarsens to 6 x 5 x 3)
        _single("box96x80x48_mixed", (48, 80, 96), 1, 3, "bubbles", 0.05, 0.05, 2.0, 0.005),
        # the 3D bubbles in both forms
        _single("bubbles128_f64", (128, 128, 128), 0, 2, "bubbles", 0.05, 0.04, 2.0, 0.005),
        _single("bubbles128_mixed", (128, 128, 128), 1, 3, "bubbles", 0.05, 0.04, 2.0, 0.005),
        # the largest 3D run of the serving stream
        _single("bubbles256_mixed", (256, 256, 256), 1, 1, "bubbles", 0.05, 0.04, 2.0, 0.005),
        # many runs of uneven size stepped together
        dict(name="batch24", kind="batch", runs=24, largest=1024, pick=4, steps=2, dt=0.005),
        # short requests through the request loop, from host fields
        dict(name="served6", kind="server", runs=6, largest=512, pick=5, steps=6, dt=0.005),
    ]


def draw(rng):
    kind = rng.choices(("2d", "3d", "batch", "server"), (5, 4, 1, 1))[0]
    if kind == "batch":
        return dict(kind="batch", runs=rng.randint(3, 24), largest=rng.choice((128, 256, 512, 1024)),
                    pick=rng.randint(1, 9999), steps=rng.randint(1, 2), dt=0.005)
    if kind == "server":
        return dict(kind="server", runs=rng.randint(2, 6), largest=rng.choice((128, 256, 512)),
                    pick=rng.randint(1, 9999), steps=rng.randint(3, 6), dt=0.005)
    precision = rng.randint(0, 1)
    if kind == "2d":
        # sides m 2^k with a small odd or even m: the grid coarsens to a few cells
        top = 2048 if precision else 1024
        side = lambda: _side(rng, 32, top, (2, 2, 2, 3, 3, 5, 6, 7, 9))
        (mx, kx), (my, ky) = side(), side()
        k = max(kx, ky) if rng.random() < 0.5 else kx
        shape = _levelled([(my, ky), (mx, kx)], k, 32, top)
        h = rng.choice((0.0125, 0.025, 0.05))
        field = rng.choice(("noise", "domains"))
    else:
        top = 256 if precision else 128
        side = lambda: _side(rng, 16, top, (2, 2, 3, 3, 4, 5))
        sides = [side() for _ in range(3)]
        shape = _levelled(sides, sides[0][1], 16, top)
        h = 0.05
        field = "bubbles"
    cells = math.prod(shape)
    steps = max(1, min(4, (1 << 20) // cells))
    eps = round(h * rng.uniform(0.8, 2.4), 4)
    gamma = rng.choice((0.0, 0.5, 1.0, 2.0, round(rng.uniform(0.5, 4.0), 2)))
    return _single(None, shape, precision, steps, field, h, eps, gamma, rng.choice((0.005, 0.01)),
                   diagnostics=rng.random() < 0.25)


def _single(name, shape, precision, steps, field, h, eps, gamma, dt, diagnostics=False):
    c = dict(kind="run", nz=shape[0] if len(shape) == 3 else 0, ny=shape[-2], nx=shape[-1], precision=precision,
             steps=steps, field=field, h=h, eps=eps, gamma=gamma, dt=dt, diagnostics=diagnostics)
    return dict(c, name=name) if name else c


def _side(rng, lo, hi, odds):
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    m = rng.choice(odds)
    return m, max(0, round(math.log2(n / m)))


def _levelled(sides, k, lo, hi):
    """Sides m 2^k with one k for all of them, each kept within [lo, hi]."""
    while any(m << k > hi for m, _ in sides):
        k -= 1
    while any(m << k < lo for m, _ in sides) and all(m << (k + 1) <= hi for m, _ in sides):
        k += 1
    return tuple(m << k for m, _ in sides)


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _noise(shape, g, mean):
    r = torch.rand(shape, generator=g, dtype=torch.float64, device=g.device)
    return mean + 0.05 * (2.0 * r - 1.0)


def _domains(shape, h, eps, g):
    """(phi, phi_prev): tanh profiles across the zero lines of a smooth random
    field (cosine modes, so that it meets the Neumann walls), the lines of the
    level before moved by a small part of the interface's width."""
    dev = g.device
    basis = []
    for n in shape:
        modes = max(3, min(24, round(n * h / (14.0 * eps))))
        x = (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) / n
        basis.append(torch.cos(math.pi * torch.arange(modes, dtype=torch.float64, device=dev)[:, None] * x))

    def smooth():
        a = torch.randn([b.shape[0] for b in basis], generator=g, dtype=torch.float64, device=dev)
        for b in basis:
            a = torch.tensordot(a, b, dims=([0], [0]))
        return a / a.square().mean().sqrt()

    f, w = smooth(), smooth()
    slope = math.sqrt(sum(float(f.diff(dim=d).square().mean()) for d in range(f.dim()))) / h
    scale = math.sqrt(2.0) * eps * slope
    return torch.tanh(f / scale).contiguous(), torch.tanh((f + 0.02 * eps * slope * w) / scale).contiguous()


def _bubbles(shape, h, eps, g):
    """Eight tanh spheres on phi = -1, sized to the box."""
    dev = g.device
    ext = [n * h for n in shape]
    u = torch.rand((8, 4), generator=g, dtype=torch.float64, device=dev).tolist()
    x = [(torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * h for n in shape]
    phi = torch.full(tuple(shape), -1.0, dtype=torch.float64, device=dev)
    for row in u:
        radius = min(ext) * (0.08 + 0.08 * row[0])
        d2 = 0.0
        for a, e in enumerate(ext):
            c = radius + (e - 2.0 * radius) * row[1 + a]
            d2 = d2 + ((x[a] - c) ** 2).reshape([-1 if b == a else 1 for b in range(len(ext))])
        phi = torch.maximum(phi, torch.tanh((radius - d2.sqrt()) / (math.sqrt(2.0) * eps)))
    return phi.contiguous()


def _fields(field, shape, h, eps, seed):
    """(phi^0, phi^{-1}); the second is None at the start of a run."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    if field == "noise":
        return _noise(shape, g, -0.05), None
    if field == "bubbles":
        return _bubbles(shape, h, eps, g), None
    return _domains(shape, h, eps, g)


def _shape(case):
    return ((case["nz"],) if case["nz"] else ()) + (case["ny"], case["nx"])


def _mix(case):
    """The runs of a batch or a stream: (shape, field, h, eps, gamma)."""
    rng = random.Random(case["pick"])
    runs = []
    for k in range(case["runs"]):
        eps, gamma = rng.uniform(0.02, 0.08), rng.uniform(0.5, 4.0)
        if case["kind"] == "server" and k % 3 == 2:
            runs.append(((64, 64, 64), "bubbles", 0.05, eps, gamma))
        else:
            lo = 64 if case["kind"] == "batch" else 128
            n = case["largest"] if k == 0 else rng.choice([s for s in (64, 128, 256, 512, 1024) if lo <= s <= case["largest"]])
            runs.append(((n, n), "noise", 0.025, eps, gamma))
    return runs


def prepare(case, seed):
    if case["kind"] == "server":
        jobs = []
        for k, (shape, field, h, eps, gamma) in enumerate(_mix(case)):
            phi, _ = _fields(field, shape, h, eps, seed * 1000 + k)
            jobs.append((shape, h, eps, gamma, case["dt"], case["steps"], phi.cpu().numpy()))
        return dict(case=case, jobs=jobs, server=chhs.Server(pool_bytes=4 << 30, max_active=12, steps_per_slice=5))
    stream = torch.cuda.Stream()
    if case["kind"] == "batch":
        mix = _mix(case)
        phis = [_fields(field, shape, h, eps, seed * 1000 + k)[0] for k, (shape, field, h, eps, _) in enumerate(mix)]
        torch.cuda.synchronize()
        batch = chhs.Batch([(shape, h, eps, gamma, case["dt"]) for shape, _, h, eps, gamma in mix],
                           stream=stream.cuda_stream)
        return dict(case=case, stream=stream, batch=batch, phis=phis, outs=[_outputs(p) for p in phis])
    shape = _shape(case)
    phi, prev = _fields(case["field"], shape, case["h"], case["eps"], seed)
    torch.cuda.synchronize()
    run = chhs.Run(shape, case["h"], case["eps"], case["gamma"], case["dt"],
                   opts=chhs.default_opts(precision=case["precision"]), stream=stream.cuda_stream)
    return dict(case=case, stream=stream, run=run, phi=phi, prev=prev, out=_outputs(phi))


def _outputs(phi):
    return {k: torch.empty_like(phi) for k in ("phi", "phi_prev", "mu", "p")}


def _read(run, out):
    """The run's state into the caller's device arrays (chhs_get_state)."""
    s = chhs.lib().chhs_get_state(run.handle, *[out[k].data_ptr() for k in ("phi", "phi_prev", "mu", "p")], 1)
    if s != chhs.CHHS_OK:
        raise chhs.ChhsError(s, "chhs_get_state failed")
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "server":
        sv = state["server"]
        ids = [sv.submit(*job, precision=1) for job in state["jobs"]]
        fields = []
        for i in ids:
            sv.wait(i)
            r = sv.result(i)
            if not r["done"] or r["status"] != chhs.CHHS_OK:
                raise RuntimeError("request %d did not converge" % i)
            fields.append(r["phi"])
            sv.release(i)
        return fields
    if case["kind"] == "batch":
        b = state["batch"]
        for r, phi in zip(b.runs, state["phis"]):
            r.set_phi(phi)
        b.step(case["steps"])
        return [_read(r, out) for r, out in zip(b.runs, state["outs"])][:: max(1, len(b.runs) // 8)]
    r = state["run"]
    r.set_phi(state["phi"], state["prev"])
    if not case["diagnostics"]:
        r.step(case["steps"])
        return _read(r, state["out"])
    rows = []
    for _ in range(case["steps"]):
        r.step(1)
        energy, modified = r.energy()
        grad_mu, u_sq, _ = r.dissipation()  # the third is the solver's own residual of div u = 0
        rows.append([energy, modified, r.mass(), grad_mu, u_sq])
    return dict(_read(r, state["out"]), rows=np.array(rows))


# ------------------------------------------------------------------ work

def _cell_steps(case):
    if case["kind"] == "run":
        return math.prod(_shape(case)) * case["steps"], math.prod(_shape(case))
    cells = sum(math.prod(m[0]) for m in _mix(case))
    return cells * case["steps"], cells


def work(case):
    """Bytes: the starting fields read and the state written once.  Operations:
    about eight V(2,2) cycles bring a step to 1e-10; a cycle is four updates and
    a residual of some 70 operations for every cell, a third of that again on
    the coarser levels in 2D and a seventh in 3D."""
    cell_steps, cells = _cell_steps(case)
    three = case["kind"] == "run" and case["nz"]
    return dict(bytes=8.0 * cells * (6 if case.get("field") == "domains" else 5 if case["kind"] != "server" else 2),
                flops=cell_steps * 8 * 5 * 70.0 * (8.0 / 7.0 if three else 4.0 / 3.0))


# ------------------------------------------------------------------ 64-bit values

def _dct(x, d):
    """DCT-II along dimension d through one complex transform of the same length."""
    n = x.shape[d]
    v = torch.cat([x.narrow(d, 0, n).index_select(d, torch.arange(0, n, 2, device=x.device)),
                   x.index_select(d, torch.arange(1, n, 2, device=x.device)).flip(d)], dim=d)
    k = torch.arange(n, dtype=torch.float64, device=x.device) * (-math.pi / (2 * n))
    w = torch.complex(torch.cos(k), torch.sin(k)).reshape([-1 if a == d else 1 for a in range(x.dim())])
    return (torch.fft.fft(v, dim=d) * w).real * 2.0


def _idct(X, d):
    n = X.shape[d]
    k = torch.arange(n, dtype=torch.float64, device=X.device) * (math.pi / (2 * n))
    w = torch.complex(torch.cos(k), torch.sin(k)).reshape([-1 if a == d else 1 for a in range(X.dim())])
    tail = torch.cat([torch.zeros_like(X.narrow(d, 0, 1)), X.narrow(d, 1, n - 1).flip(d)], dim=d)
    v = torch.fft.ifft(0.5 * w * torch.complex(X, -tail), dim=d).real
    x = torch.empty_like(X)
    half = (n + 1) // 2
    even = torch.arange(0, n, 2, device=X.device)
    odd = torch.arange(1, n, 2, device=X.device)
    x.index_copy_(d, even, v.narrow(d, 0, half))
    if n > 1:
        x.index_copy_(d, odd, v.narrow(d, half, n - half).flip(d))
    return x


class _Scheme:
    """A step of the scheme solved in 64 bits: p is eliminated by cosine
    transforms, phi found by Newton's method with GMRES."""

    def __init__(self, shape, h, eps, gamma, dt, dev):
        self.shape, self.h, self.eps, self.gamma, self.s, self.dim = shape, h, eps, gamma, dt, len(shape)
        lam = torch.zeros(shape, dtype=torch.float64, device=dev)
        for d, n in enumerate(shape):
            k = torch.arange(n, dtype=torch.float64, device=dev)
            lam = lam + (-4.0 / h**2 * torch.sin(0.5 * math.pi * k / n) ** 2).reshape([-1 if a == d else 1 for a in range(len(shape))])
        self.lam = lam
        inv = lam.clone()
        inv.view(-1)[0] = 1.0
        self.inv_lam = 1.0 / inv
        self.inv_lam.view(-1)[0] = 0.0

    def spectral(self, x, factor):
        for d in range(self.dim):
            x = _dct(x, d)
        x = x * factor
        for d in range(self.dim):
            x = _idct(x, d)
        return x

    def div(self, u, faces=None):
        """div(c grad u) with the face values c (1 if None), no flux through the walls."""
        out = torch.zeros_like(u)
        for d, n in enumerate(self.shape):
            f = u.diff(dim=d) / self.h**2
            if faces is not None:
                f = faces[d] * f
            out.narrow(d, 0, n - 1).add_(f)
            out.narrow(d, 1, n - 1).sub_(f)
        return out

    def average(self, u):
        return [0.5 * (u.narrow(d, 0, n - 1) + u.narrow(d, 1, n - 1)) for d, n in enumerate(self.shape)]

    def pressure(self, mu):
        return self.spectral(self.div(mu, self.a), -self.gamma * self.inv_lam)

    def flow(self, mu):
        return self.div(mu, self.M) + self.div(self.pressure(mu), self.a)

    def gmres(self, apply, precondition, b, target, most=60):
        beta = float(b.norm())
        basis, hess = [b / beta], np.zeros((most + 1, most))
        for j in range(most):
            w = apply(precondition(basis[j]))
            for _ in range(2):
                for i in range(j + 1):
                    c = float(torch.vdot(basis[i].reshape(-1), w.reshape(-1)))
                    hess[i, j] += c
                    w = w - c * basis[i]
            hess[j + 1, j] = float(w.norm())
            rhs = np.zeros(j + 2)
            rhs[0] = beta
            y = np.linalg.lstsq(hess[: j + 2, : j + 1], rhs, rcond=None)[0]
            if np.linalg.norm(hess[: j + 2, : j + 1] @ y - rhs) <= target * beta or hess[j + 1, j] <= 1e-300:
                break
            basis.append(w / hess[j + 1, j])
        return precondition(sum(float(c) * v for c, v in zip(y, basis)))

    def step(self, phim, prev):
        star = 1.5 * phim - 0.5 * prev
        self.a = self.average(star)
        self.M = [1.0 + self.gamma * a * a for a in self.a]
        fixed = star + 0.25 * self.eps**2 * self.div(prev)

        def mu_of(phi):
            return 0.25 * (phi * phi + phim * phim) * (phi + phim) - fixed - 0.75 * self.eps**2 * self.div(phi)

        kappa = 1.0 + self.gamma * float(star.square().mean()) * (self.dim - 1) / self.dim
        phi = 2.0 * phim - prev
        last = math.inf
        for _ in range(12):
            mu = mu_of(phi)
            r = phi - phim - self.s * self.flow(mu)
            size = float(r.square().mean().sqrt())
            if size < 2e-15 or (size < 1e-11 and size > 0.5 * last):
                break
            last = size
            slope = 0.25 * (3.0 * phi * phi + 2.0 * phi * phim + phim * phim)
            c = float(slope.mean())
            pre = 1.0 / (1.0 - self.s * kappa * self.lam * (c - 0.75 * self.eps**2 * self.lam))
            d = self.gmres(lambda v: v - self.s * self.flow(slope * v - 0.75 * self.eps**2 * self.div(v)),
                           lambda v: self.spectral(v, pre), -r, 1e-5 if size > 1e-9 else 1e-3)
            phi = phi + d
        mu = mu_of(phi)
        return phi, mu, self.pressure(mu)

    def rows(self, phi, prev, mu, p):
        cell = self.h**self.dim

        def energy(f):
            return (0.25 * float((f**4).sum()) - 0.5 * float((f * f).sum())) * cell + 0.5 * self.eps**2 * grad(f)

        def grad(f):
            return cell * sum(float((f.diff(dim=d) / self.h).square().sum()) for d in range(self.dim))

        e = energy(phi)
        d = phi - prev
        u_sq = cell * sum(float((p.diff(dim=k) / self.h + self.gamma * self.a[k] * mu.diff(dim=k) / self.h).square().sum())
                          for k in range(self.dim))
        return [e, e + 0.25 * cell * float((d * d).sum()) + 0.125 * self.eps**2 * grad(d), cell * float(phi.sum()),
                grad(mu), u_sq]


def exact(case, seed):
    if case["kind"] == "run":
        shape = _shape(case)
        if math.prod(shape) * case["steps"] > 9 << 20:
            return None
        phi, prev = _fields(case["field"], shape, case["h"], case["eps"], seed)
        return _exact_run(shape, case["h"], case["eps"], case["gamma"], case["dt"], case["steps"], phi, prev,
                          case["diagnostics"])
    out = []
    for k, (shape, field, h, eps, gamma) in enumerate(_mix(case)):
        if case["kind"] == "batch" and k % max(1, case["runs"] // 8):
            continue
        phi, prev = _fields(field, shape, h, eps, seed * 1000 + k)
        got = _exact_run(shape, h, eps, gamma, case["dt"], case["steps"], phi, prev, False)
        out.append(got["phi"].cpu().numpy() if case["kind"] == "server" else got)
    return out


def _exact_run(shape, h, eps, gamma, dt, steps, phi, prev, diagnostics):
    scheme = _Scheme(shape, h, eps, gamma, dt, phi.device)
    prev = phi if prev is None else prev
    rows = []
    for _ in range(steps):
        new, mu, p = scheme.step(phi, prev)
        phi, prev = new, phi
        if diagnostics:
            rows.append(scheme.rows(phi, prev, mu, p))
    out = dict(phi=phi, phi_prev=prev, mu=mu, p=p)
    return dict(out, rows=np.array(rows)) if diagnostics else out
