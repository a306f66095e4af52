"""The work that a user of the library has it do, as cases with sizes.

A pass is one whole call sequence of a user's program: give the initial phase
fields to a simulation (or an ensemble) that the program keeps, advance it,
read the moments; or one gradient evaluation of a loss of the final fields.
The passes are short (6 to 40 steps): the method amplifies rounding by itself,
and a longer run says nothing about what a pass computed.

``exact`` is the same computation in 64 bits, written with torch operations
from the method's equations (arXiv 2306.06983, Secs. 2-4): the phase-field and
flow populations with the moment-space collision in closed form, mirrored
stencils and half-way bounce-back at walls.
"""

from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2306_06983_gb300.nlbm import AdjointRun, Batch, Simulation, nphase_lbm

DEV = "cuda"
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def listed():
    return [
        # The three-phase droplets on 64 x 64 that the library's first checks
        # and its users' first scripts run: the smallest call, all latency.
        case("droplets 64", "sim", "disks", 64, 64, 3, steps=10),
        # The paper's Table 1: four phases at a density ratio of 1000 on its
        # 300 x 100 domain, Model A with n = 2; parameter scans run thousands
        # of such small problems.
        case("static drops 300x100", "sim", "static", 300, 100, 4, model="A", n=2.0, eps=5.0, mobility=0.01, steps=20),
        # The paper's Table 2: a compound droplet on a wetting wall.
        case("wetting 300x150", "sim", "compound", 300, 150, 3, eps=5.0, wall_y=True, wet=True, steps=20),
        # The paper's Rayleigh-Taylor instability: walls, gravity, a lattice
        # of ordinary size.
        case("rayleigh-taylor 256x1024", "sim", "rt", 256, 1024, 3, wall_y=True, gravity=6.25e-6, steps=20),
        # A closed box of odd size: walls on both axes, rows that start on no
        # particular boundary, a non-integer Model A exponent.
        case("closed box 509x383", "sim", "disks", 509, 383, 4, model="A", n=1.5, wall_x=True, wall_y=True, steps=10),
        # Eight phases, the most that the library takes, Model A.
        case("eight phases 1024", "sim", "disks", 1024, 1024, 8, model="A", n=1.0, steps=10),
        # The headline workload: a five-phase suspension on 2048 x 2048, with
        # the tile that the library's tuner picks (as long runs do).
        case("suspension 2048", "sim", "disks", 2048, 2048, 5, tuned=True, steps=10),
        # The same with bfloat16 populations, for lattices where memory counts.
        case("suspension 2048 bf16", "sim", "disks", 2048, 2048, 5, storage="bf16", tuned=True, steps=10),
        # binary16 populations on an ordinary lattice, an odd number of solved
        # phases (an unpaired 16-bit plane), Model A, the library's own tile.
        case("suspension 504x376 f16", "sim", "disks", 504, 376, 4, model="A", n=1.0, storage="f16", steps=20),
        # A sweep over 64 independent lens problems of three sizes, both
        # models, advanced together (the paper's Table 3 done as one run).
        case("lens ensemble 64", "batch", "lens", 512, 256, 3, count=64, wall_y=True, tuned=True, steps=32),
        # The gradient study on 256 x 256 through a handle that an optimiser
        # keeps: forward with checkpoints, then the reverse sweep.
        case("gradient 256", "handle", "disks", 256, 256, 3, delta=1e-3, every=20, steps=40),
        # The same problem on 1024 x 1024 through torch.autograd.
        case("gradient 1024 autograd", "autograd", "disks", 1024, 1024, 3, delta=1e-3, every=8, steps=16),
    ]


def case(name, form, field, nx, ny, N, model="B", n=1.0, eps=4.0, mobility=0.1, storage="f32", wall_x=False,
         wall_y=False, wet=False, gravity=0.0, delta=0.0, tuned=False, count=1, every=0, steps=20):
    c = dict(form=form, field=field, nx=nx, ny=ny, N=N, model=model, n=n, eps=eps, mobility=mobility, storage=storage,
             wall_x=wall_x, wall_y=wall_y, wet=wet, gravity=gravity, delta=delta, tuned=tuned, count=count,
             every=every, steps=steps)
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choices(("sim", "sim16", "batch", "handle", "autograd"), (9, 3, 2, 2, 1))[0]
    model = rng.choice("AB")
    n = rng.choice((0.5, 1.0, 1.0, 2.0, 3.0)) if model == "A" else 1.0
    if form in ("handle", "autograd"):
        # Gradient runs: three phases mostly, smooth unit vectors, periodic or walls.
        N = rng.choice((2, 3, 3, 4))
        nx = _log(rng, 48, 1024)
        ny = max(48, min(1024, int(nx * rng.uniform(0.5, 1.5))))
        steps = rng.randint(8, 16) if nx * ny > 300000 else rng.randint(12, 40)
        return case(None, form, "disks", nx, ny, N, model=model, n=max(n, 1.0), wall_x=rng.random() < 0.15,
                    wall_y=rng.random() < 0.25, delta=1e-3, every=rng.choice((5, 8, 10, 20)), steps=steps)
    if form == "batch":
        # Ensembles share N; members keep the case's model with walls on y.
        return case(None, "batch", "lens", 32 * rng.randint(4, 16), 16 * rng.randint(4, 16), 3, model=model, n=n,
                    count=rng.randint(2, 48), wall_y=True, tuned=rng.random() < 0.5, steps=rng.randint(8, 24))
    N = rng.choice((2, 3, 3, 4, 5, 5, 6, 7, 8))
    side = _log(rng, 40, 2048)
    nx = max(32, int(side * math.sqrt(rng.uniform(0.5, 2.0))))
    ny = max(32, min(4096, side * side // nx))
    while nx * ny * (10 * N + 2) > 2048 * 2048 * 52:
        N = max(2, N - 1)
        ny = min(ny, 2048 * 2048 * 52 // (nx * (10 * N + 2)))
    if form == "sim16":
        nx += nx % 2 if rng.random() < 0.5 else -nx % 8
        ny = min(ny, 2048 * 2048 * 52 // (nx * (10 * N + 2)))
        return case(None, "sim", "disks", nx, ny, N, model=model, n=n, storage=rng.choice(("bf16", "f16")),
                    wall_y=rng.random() < 0.25, tuned=nx * ny > 500000 and rng.random() < 0.5, steps=rng.randint(6, 10))
    r = rng.random()
    wall_x, wall_y = r < 0.15, 0.08 < r < 0.4
    if rng.random() < 0.6:
        nx += -nx % 4
        ny = min(ny, 2048 * 2048 * 52 // (nx * (10 * N + 2)))
    return case(None, "sim", "disks", nx, ny, N, model=model, n=n, eps=rng.choice((4.0, 4.0, 5.0)), wall_x=wall_x,
                wall_y=wall_y, wet=wall_y and rng.random() < 0.3, gravity=6.25e-6 if rng.random() < 0.3 else 0.0,
                tuned=nx * ny > 500000 and rng.random() < 0.5, steps=rng.randint(6, 10))


# ------------------------------------------------------------------ problems

def _problem(c, rng, nx, ny, model, n):
    """(parameters, phases 1..N-1 as a float32 CUDA tensor) of one simulation."""
    N, eps = c["N"], c["eps"]
    rho = np.array([1.0, 2.0, 5.0, 10.0, 1.0, 3.0, 7.0, 4.0])[:N]
    mu = rho * rng.uniform(0.02, 0.1, N)
    sig = np.zeros((N, N))
    for a in range(N):
        for b in range(a + 1, N):
            sig[a, b] = sig[b, a] = rng.uniform(0.005, 0.02)
    x = torch.arange(nx, dtype=torch.float64, device=DEV)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=DEV)[:, None]
    wall_cos, gy = None, -c["gravity"]

    def step(d, width):
        return 0.5 + 0.5 * torch.tanh(d / width)

    if c["field"] == "static":
        rho = np.array([1000.0, 500.0, 100.0, 1.0])
        mu = 0.1 * rho
        phi = torch.stack([step(20.0 + rng.uniform(-2, 2) - torch.hypot(x - cx, y - (ny / 2.0 + rng.uniform(-5, 5))), eps / 2)
                           for cx in nx * (np.arange(N - 1) + 0.5) / (N - 1) + rng.uniform(-5, 5, N - 1)])
    elif c["field"] == "compound":
        rho, mu = np.array([1.0, 0.5, 0.001]), np.array([0.1, 0.05, 1e-4])
        cx, R = nx / 2.0 + rng.uniform(-10, 10), 60.0 * ny / 150.0 * rng.uniform(0.9, 1.1)
        D = step(R - torch.hypot(x - cx, y + 0.5), eps / 2)
        phi = torch.stack([D * step(cx - x + 0 * y, eps / 2), D * step(x - cx + 0 * y, eps / 2)])
        wall_cos = [math.cos(math.radians(75.0)), math.cos(math.radians(rng.uniform(40, 110))), 0.0, 0.0]
    elif c["field"] == "rt":
        rho, mu = np.array([3.0, 2.0, 1.0]), np.full(3, 0.01024)
        sig = np.full((3, 3), 1.46e-3) * (1 - np.eye(3))
        s = 0.1 * nx * torch.sin(2 * math.pi * x / nx + rng.uniform(0, 6.28))
        phi1 = step(y - 2 * ny / 3.0 - s, eps / 2)
        phi = torch.stack([phi1, (1 - phi1) * step(y - ny / 3.0 + s, eps / 2)])
    elif c["field"] == "lens":
        rho, mu = np.ones(3), np.full(3, 1.0 / 6.0)
        s13, s23 = rng.uniform(0.005, 0.015, 2)
        sig = np.array([[0, 0.01, s13], [0.01, 0, s23], [s13, s23, 0]])
        L = step(0.2 * ny - torch.hypot(x - nx / 2.0, y - (ny / 2.0 - 0.5)), eps / 2)
        B = step(ny / 2.0 - 0.5 - y + 0 * x, eps / 2)
        phi = torch.stack([(1 - L) * B, (1 - L) * (1 - B)])
    else:   # non-overlapping disks of phases 2..N in a matrix of phase 1
        R0 = max(7.0, min(40.0, min(nx, ny) / 12.0)) + eps
        kx, ky = max(1, int(nx / (2.6 * R0))), max(1, int(ny / (2.6 * R0)))
        phi = torch.zeros((N, ny, nx), dtype=torch.float64, device=DEV)
        for k in rng.permutation(kx * ky)[: max(2, min(200, 2 * kx * ky // 3))]:
            R = (R0 - eps) * rng.uniform(0.55, 1.0)
            cx, cy = (k % kx + 0.5) * nx / kx + rng.uniform(-2, 2), (k // kx + 0.5) * ny / ky + rng.uniform(-2, 2)
            x0, x1 = max(0, int(cx - R - 10 * eps)), min(nx, int(cx + R + 10 * eps))
            y0, y1 = max(0, int(cy - R - 10 * eps)), min(ny, int(cy + R + 10 * eps))
            phi[rng.integers(1, N), y0:y1, x0:x1] += step(R - torch.hypot(x[:, x0:x1] - cx, y[y0:y1] - cy), eps / 2)
        phi[0] = 1 - phi[1:].sum(0)
        phi = phi[: N - 1]
    if c["wet"] and wall_cos is None:
        wall_cos = [float(v) for v in np.cos(np.radians(rng.uniform(60, 120, 2 * (N - 1))))]
        wall_cos[: N - 2] = wall_cos[N - 1: 2 * N - 3] = [0.0] * (N - 2)   # the last solved phase alone wets
    p = dict(nx=nx, ny=ny, n_phases=N, model=model, model_a_n=n, eps=eps, mobility=c["mobility"], rho=rho.tolist(),
             mu=mu.tolist(), sigma=sig.tolist(), wall_x=c["wall_x"], wall_y=c["wall_y"], storage=c["storage"],
             unit_delta=c["delta"], gx=0.0, gy=gy, wall_cos=wall_cos)
    return p, phi.float().contiguous()


def _members(c, rng):
    """An ensemble's members: lattices of the case's size, half and a quarter
    of it in turn, the first half Model B, the second half Model A with its exponent
    swept; or all of the case's own model, where that is Model A."""
    out = []
    for k in range(c["count"]):
        nx, ny = c["nx"] >> k % 3, c["ny"] >> k % 3
        a = c["model"] == "A" or k >= c["count"] // 2
        out.append(_problem(c, rng, nx, ny, "A" if a else "B", c["n"] if c["model"] == "A" else 0.5 + 0.5 * (k % 8)))
    return out


def _gradient_problem(c, rng):
    p, phi0 = _problem(c, rng, c["nx"], c["ny"], c["model"], c["n"])
    N = c["N"]
    p = dict(p, rho=[1.0] * N, mu=[1.0 / 6.0] * N)
    pairs = [(a, b) for a in range(N) for b in range(a + 1, N)]
    sig = np.array([p["sigma"][a][b] for a, b in pairs], dtype=np.float32)
    full = torch.cat([phi0, 1 - phi0.sum(0, keepdim=True)])
    return p, phi0, pairs, sig, torch.roll(full, (3, 2), (1, 2)).contiguous()


def _rng(seed):
    return np.random.default_rng([2306, int(seed)])


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    c, rng = case, _rng(seed)
    if c["form"] == "sim":
        p, phi0 = _problem(c, rng, c["nx"], c["ny"], c["model"], c["n"])
        sim = Simulation(p)
        if c["tuned"]:
            sim.set_phi(phi0)
            sim.autotune()
        return dict(case=c, sim=sim, phi0=phi0)
    # ensembles and gradient handles live on a stream of their own, where
    # their launches can be replayed as graphs
    if c["form"] == "batch":
        mem = _members(c, rng)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            b = Batch([p for p, _ in mem])
            if c["tuned"]:
                for k, (_, f) in enumerate(mem):
                    b.set_phi(k, f)
                b.autotune()
        return dict(case=c, batch=b, stream=stream, phi0=[f for _, f in mem])
    p, phi0, pairs, sig, target = _gradient_problem(c, rng)
    if c["form"] == "autograd":
        return dict(case=c, params=p, phi0=phi0, sigma=torch.from_numpy(sig), mobility=torch.tensor(c["mobility"]), target=target)
    for (a, b), v in zip(pairs, sig):
        p["sigma"][a][b] = p["sigma"][b][a] = float(v)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        run_ = AdjointRun(p, c["steps"], c["every"])
    return dict(case=c, run=run_, stream=stream, phi0=phi0, target=target, pairs=pairs)


def run(state):
    c = state["case"]
    if c["form"] == "sim":
        sim = state["sim"]
        sim.set_phi(state["phi0"])
        sim.step(c["steps"])
        return dict(zip(("phi", "u", "p"), sim.moments()))
    if c["form"] == "autograd":
        phi0 = state["phi0"].clone().requires_grad_()
        sigma = state["sigma"].clone().requires_grad_()
        mobility = state["mobility"].clone().requires_grad_()
        phi = nphase_lbm(phi0, sigma, mobility, state["params"], c["steps"], c["every"])
        (0.5 * (phi - state["target"]).square().sum()).backward()
        return dict(phi=phi.detach(), phi0=phi0.grad, sigma=sigma.grad, mobility=mobility.grad)
    stream = state["stream"]
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        if c["form"] == "batch":
            b = state["batch"]
            for k, f in enumerate(state["phi0"]):
                b.set_phi(k, f)
            b.step(c["steps"])
            m = [b.moments(k) for k in range(len(b))]
            out = {name: torch.cat([v[j].reshape(-1) for v in m]) for j, name in enumerate(("phi", "u", "p"))}
        else:
            phi = state["run"].forward(state["phi0"])
            g0, gs, gm = state["run"].backward(phi - state["target"])
            out = dict(phi=phi, phi0=g0, mobility=gm,   # the optimiser holds the tensions in 32 bits
                       sigma=torch.tensor([gs[a, b] for a, b in state["pairs"]], dtype=torch.float32))
    torch.cuda.current_stream().wait_stream(stream)
    return out


# ------------------------------------------------------------------ floors

def work(case):
    c, N = case, case["N"]
    nodes = c["nx"] * c["ny"]
    if c["form"] == "batch":
        nodes *= c["count"] * (1 + 1 / 4 + 1 / 16) / 3   # members of three sizes
    # every stored value read once and written once a step: 9 (N-1) + 8
    # populations, N-1 phase fields, u and m_phi; in 16 bits the 8 moving
    # populations of each set, with the rest populations and the pressure in 32
    update = 8 * (10 * N + 2) if c["storage"] == "f32" else 48 * (N - 1) + 72
    flops = 300 + 130 * (N - 1) + 45 * N * (N - 1) / 2
    ends = 4 * (N - 1) + 4 * (N + 3)
    if c["form"] in ("handle", "autograd"):
        # the reverse needs each step's state again (rebuilt: one update), and
        # reads and writes the adjoint of a state a step
        state = 4 * (10 * (N - 1) + 12)
        return dict(bytes=nodes * (c["steps"] * (2 * update + 3 * state) + ends + 8 * N), flops=nodes * c["steps"] * 5 * flops)
    return dict(bytes=nodes * (c["steps"] * update + ends), flops=nodes * c["steps"] * flops)


# ------------------------------------------------------------------ 64 bits

def _axis(n, wall):
    i = torch.arange(-2, n + 2, device=DEV)
    if wall:
        flip = (i < 0) | (i >= n)
        return torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i)), flip
    return i % n, torch.zeros_like(i, dtype=torch.bool)


def _grad(a):
    """Isotropic central gradient and Laplacian on the inside of a."""
    def s(dx, dy):
        return a[..., 1 + dy: a.shape[-2] - 1 + dy, 1 + dx: a.shape[-1] - 1 + dx]
    gx = (s(1, 0) - s(-1, 0)) / 3 + (s(1, 1) - s(-1, 1) + s(1, -1) - s(-1, -1)) / 12
    gy = (s(0, 1) - s(0, -1)) / 3 + (s(1, 1) - s(1, -1) + s(-1, 1) - s(-1, -1)) / 12
    ax = s(1, 0) + s(-1, 0) + s(0, 1) + s(0, -1)
    dg = s(1, 1) + s(-1, 1) + s(1, -1) + s(-1, -1)
    return gx, gy, 2 * ax / 3 + dg / 6 - 10 * s(0, 0) / 3


def _dot(c, a):
    return sum(v * x for v, x in zip(c, a))


class _Exact:
    """The method in 64 bits; a state is (f [N-1,9], g [9], phi, u, m_phi)."""

    def __init__(self, p):
        self.p, self.N = p, p["n_phases"]
        self.rho, self.mu = p["rho"], p["mu"]
        self.yi, self.yf = _axis(p["ny"], p["wall_y"])
        self.xi, self.xf = _axis(p["nx"], p["wall_x"])
        sgn = torch.ones((len(self.yi), len(self.xi)), dtype=torch.float64, device=DEV)
        self.usign = sgn - 2 * (self.yf[:, None] != self.xf[None, :])
        N, nx, ny = self.N, p["nx"], p["ny"]
        x, y = torch.arange(nx, device=DEV)[None, :], torch.arange(ny, device=DEV)[:, None]
        self.bounce = []
        for cx, cy in zip(CX, CY):
            m = torch.zeros((ny, nx), dtype=torch.bool, device=DEV)
            if p["wall_x"]:
                m = m | (x - cx < 0) | (x - cx >= nx)
            if p["wall_y"]:
                m = m | (y - cy < 0) | (y - cy >= ny)
            self.bounce.append(m)
        self.wet = [None, None]
        if p["wall_cos"] is not None:
            for w in range(2):
                cn = p["wall_cos"][w * (N - 1): (w + 1) * (N - 1)] + [0.0]
                s = p["sigma"]
                t = [[0.0 if a == b else cn[a] if b == N - 1 else -cn[b] if a == N - 1 else
                      (s[a][N - 1] * cn[a] - s[b][N - 1] * cn[b]) / s[a][b] for b in range(N)] for a in range(N)]
                self.wet[w] = [[4.0 / p["eps"] * v for v in r] for r in t]

    def start(self, phi0):
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        wc = torch.tensor(w, dtype=torch.float64, device=DEV)[None, :, None, None]
        z = torch.zeros_like(phi0[0])
        # as pulled: the first step sees the equilibria of a fluid at rest
        return wc * phi0[:, None], torch.zeros((9,) + z.shape, dtype=torch.float64, device=DEV), phi0, torch.stack([z, z]), torch.stack([z, z])

    def pull(self, f):
        """f[..., i] streamed along c_i, bounced back at walls."""
        out = []
        for i in range(9):
            a = torch.roll(f[..., i, :, :], (CY[i], CX[i]), (-2, -1))
            m = self.bounce[i]
            out.append(torch.where(m, f[..., OPP[i], :, :], a) if i and (self.p["wall_x"] or self.p["wall_y"]) else a)
        return torch.stack(out, -3)

    def unit(self, vx, vy):
        n2, d = vx * vx + vy * vy, self.p["unit_delta"]
        if d > 0:
            r = torch.rsqrt(n2 + d * d)
        else:
            r = torch.where(n2 > 1e-24, torch.rsqrt(torch.clamp(n2, min=1e-300)), torch.zeros_like(n2))
        return r

    def source(self, ph, gx, gy):
        N, k = self.N, 4.0 / self.p["eps"]
        if self.p["model"] == "A":
            a = [k * ph[q] * (1 - ph[q]) * self.unit(gx[q], gy[q]) for q in range(N)]
            ax, ay = [a[q] * gx[q] for q in range(N)], [a[q] * gy[q] for q in range(N)]
            w = [torch.relu(ph[q]) ** self.p["model_a_n"] for q in range(N)]
            S, Vx, Vy = sum(w), sum(ax), sum(ay)
            return [ax[q] - w[q] / S * Vx for q in range(N - 1)], [ay[q] - w[q] / S * Vy for q in range(N - 1)]
        Rx, Ry = [0.0] * N, [0.0] * N
        for p in range(N):
            for q in range(p + 1, N):
                vx, vy = ph[q] * gx[p] - ph[p] * gx[q], ph[q] * gy[p] - ph[p] * gy[q]
                c = k * ph[p] * ph[q] * self.unit(vx, vy)
                Rx[p], Ry[p], Rx[q], Ry[q] = Rx[p] + c * vx, Ry[p] + c * vy, Rx[q] - c * vx, Ry[q] - c * vy
        return Rx[: N - 1], Ry[: N - 1]

    def step(self, f, g, php, up, mp, sig, M, last=False):
        """One step from the pulled populations; returns the next pulled ones,
        the fields of this step, and with `last` the moments."""
        N, P = self.N, self.p
        NS = N - 1
        drho, dmu = [r - self.rho[-1] for r in self.rho[:NS]], [m - self.mu[-1] for m in self.mu[:NS]]
        phi = f.sum(1)
        jx, jy = _dot(CX, f.unbind(1)), _dot(CY, f.unbind(1))
        # fields with two ghost layers
        rows = phi[:, self.yi]
        if any(w is not None for w in self.wet):
            full = torch.cat([rows, 1 - rows.sum(0, keepdim=True)])
            add = torch.zeros_like(rows)
            for w, ghosts in ((0, (0, 1)), (1, (P["ny"] + 2, P["ny"] + 3))):
                for r in ghosts:
                    k2 = 2 * (2 - r if w == 0 else r - P["ny"] - 1) - 1
                    add[:, r] = torch.stack([k2 * full[a, r] * _dot(self.wet[w][a], full[:, r]) for a in range(NS)])
            rows = rows + add
        ext = rows[:, :, self.xi]
        gx, gy, lap = _grad(ext)
        ph = ext[:, 1:-1, 1:-1]

        def all_n(v, c):
            return torch.cat([v, c - v.sum(0, keepdim=True)]).unbind(0)
        phN, gxN, gyN, lapN = all_n(ph, 1), all_n(gx, 0), all_n(gy, 0), all_n(lap, 0)
        Rx, Ry = self.source(phN, gxN, gyN)
        mx1 = -M * sum(d * (gxN[q] - Rx[q]) for q, d in enumerate(drho))
        my1 = -M * sum(d * (gyN[q] - Ry[q]) for q, d in enumerate(drho))
        ug = (up[:, self.yi][:, :, self.xi] * self.usign)[:, 1:-1, 1:-1]
        wx, wy, _ = _grad(mx1 * ug[1] - ug[0] * my1)

        def inner(v):
            return [a[1:-1, 1:-1] for a in v]
        phN, gxN, gyN, lapN, Rx, Ry = inner(phN), inner(gxN), inner(gyN), inner(lapN), inner(Rx), inner(Ry)
        mphx, mphy = mx1[1:-1, 1:-1], my1[1:-1, 1:-1]
        phi = phi.unbind(0)
        rho = self.rho[-1] + _dot(drho, phi)
        mu = self.mu[-1] + _dot(dmu, phi)
        grx, gry = _dot(drho, gxN[:NS]), _dot(drho, gyN[:NS])

        def dg(s):
            return 2 * s * (1 - s) * (1 - 2 * s)
        pot = [0.0] * N
        for a in range(N):
            for b in range(a + 1, N):
                be, ka = 6 * sig[a][b] / P["eps"], 0.75 * P["eps"] * sig[a][b]
                G = dg(phN[a] + phN[b])
                pot[a] = pot[a] + be * (dg(phN[a]) - G) + ka * lapN[b]
                pot[b] = pot[b] + be * (dg(phN[b]) - G) + ka * lapN[a]
        Fx = sum((pot[a] - pot[NS]) * gxN[a] for a in range(NS)) + 0.5 * wy + rho * P["gx"]
        Fy = sum((pot[a] - pot[NS]) * gyN[a] for a in range(NS)) - 0.5 * wx + rho * P["gy"]
        g = g.unbind(0)
        sg, jgx, jgy = sum(g[1:]), _dot(CX, g), _dot(CY, g)
        Pxx, Pyy = _dot([c * c for c in CX], g), _dot([c * c for c in CY], g)
        Pxy = _dot([a * b for a, b in zip(CX, CY)], g)
        ux, uy = (jgx + 0.5 * Fx) / rho, (jgy + 0.5 * Fy) / rho
        upx, upy, mpx, mpy = up[0], up[1], mp[0], mp[1]
        mx, my = rho * ux + mphx, rho * uy + mphy
        ugr = ux * grx + uy * gry
        rho_p = self.rho[-1] + _dot(drho, php.unbind(0))
        mut, mup = mx * ux + my * uy, (rho_p * upx + mpx) * upx + (rho_p * upy + mpy) * upy
        Pr = 0.6 * (sg + 0.5 * ugr - (2 / 3) * mut + (mut - mup) / 3)
        # phase-field collision
        s1 = 1.0 / (0.5 + 3 * M)
        fo = []
        for q in range(NS):
            Gx, Gy = 3 * (phi[q] * ux - php[q] * upx) + Rx[q], 3 * (phi[q] * uy - php[q] * upy) + Ry[q]
            A = (1 - s1) * jx[q] + s1 * phi[q] * ux + (1 - s1 / 2) / 3 * Gx
            B = (1 - s1) * jy[q] + s1 * phi[q] * uy + (1 - s1 / 2) / 3 * Gy
            C, D = phi[q] * uy / 3 + Gy / 18, phi[q] * ux / 3 + Gx / 18
            a, b = phi[q] / 9, phi[q] / 36
            fo.append(torch.stack([4 * a, a + (A - D) / 2, a + (B - C) / 2, a - (A - D) / 2, a - (B - C) / 2,
                                   b + (C + D) / 4, b + (C - D) / 4, b - (C + D) / 4, b - (C - D) / 4]))
        # flow collision
        s2 = 2 * rho / (6 * mu + rho)
        Qxx, Qyy, Qxy = mx * ux, my * uy, 0.5 * (mx * uy + my * ux)
        Mxx = 2 * ux * Fx + mphx * ux - mpx * upx + (2 * ux * grx + ugr) / 3
        Myy = 2 * uy * Fy + mphy * uy - mpy * upy + (2 * uy * gry + ugr) / 3
        Mxy = ux * Fy + Fx * uy + 0.5 * (mphx * uy + mphy * ux - mpx * upy - mpy * upx) + (ux * gry + grx * uy) / 3
        m1, m2 = jgx + Fx, jgy + Fy
        m3 = (1 - s2) * Pxx + s2 * (Pr + Qxx) + (1 - s2 / 2) * Mxx
        m4 = (1 - s2) * Pyy + s2 * (Pr + Qyy) + (1 - s2 / 2) * Myy
        m5 = (1 - s2) * Pxy + s2 * Qxy + (1 - s2 / 2) * Mxy
        m6, m7 = rho * uy / 3 + Fy / 6, rho * ux / 3 + Fx / 6
        m8 = (Pr + Qxx + Qyy) / 3 + (Mxx + Myy) / 6 - ugr / 18
        go = torch.stack([0 * m1, (m1 - m7 + m3 - m8) / 2, (m2 - m6 + m4 - m8) / 2, (m7 - m1 + m3 - m8) / 2,
                          (m6 - m2 + m4 - m8) / 2, (m5 + m6 + m7 + m8) / 4, (m6 - m5 + m8 - m7) / 4,
                          (m5 - m6 + m8 - m7) / 4, (m7 - m5 + m8 - m6) / 4])
        out = self.pull(torch.stack(fo)), self.pull(go), torch.stack(phi), torch.stack([ux, uy]), torch.stack([mphx, mphy])
        return out + (Pr,) if last else out


def _exact_sim(p, phi0, steps):
    e = _Exact(p)
    s = e.start(phi0.double())
    with torch.no_grad():
        for k in range(steps - 1):
            s = e.step(*s, p["sigma"], p["mobility"])
        s = e.step(*s, p["sigma"], p["mobility"], last=True)
    return torch.cat([s[2], 1 - s[2].sum(0, keepdim=True)]), s[3], s[5]


def exact(case, seed):
    c, rng = case, _rng(seed)
    if c["form"] == "sim":
        p, phi0 = _problem(c, rng, c["nx"], c["ny"], c["model"], c["n"])
        return dict(zip(("phi", "u", "p"), _exact_sim(p, phi0, c["steps"])))
    if c["form"] == "batch":
        m = [_exact_sim(p, f, c["steps"]) for p, f in _members(c, rng)]
        return {name: torch.cat([v[j].reshape(-1) for v in m]) for j, name in enumerate(("phi", "u", "p"))}
    p, phi0, pairs, sig, target = _gradient_problem(c, rng)
    N, e = c["N"], _Exact(p)
    phi0 = phi0.double().requires_grad_()
    sigma = torch.from_numpy(sig).double().to(DEV).requires_grad_()
    # the handle is given the mobility itself, autograd a 32-bit parameter
    M = torch.tensor(c["mobility"], dtype=torch.float64 if c["form"] == "handle" else torch.float32).double().to(DEV)
    M = M.requires_grad_()

    def step(f, g, ph, u, m, sigma, M):
        table = [[None] * N for _ in range(N)]
        for (a, b), v in zip(pairs, sigma.unbind(0)):
            table[a][b] = table[b][a] = v
        return e.step(f, g, ph, u, m, table, M)

    s = e.start(phi0)
    for k in range(c["steps"]):
        s = checkpoint(step, *s, sigma, M, use_reentrant=False)
    phi = torch.cat([s[2], 1 - s[2].sum(0, keepdim=True)])
    (0.5 * (phi - target.double()).square().sum()).backward()
    return dict(phi=phi.detach(), phi0=phi0.grad, sigma=sigma.grad, mobility=M.grad)
