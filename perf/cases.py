"""Cases by which the speed of the composite step is measured.

Every case is a whole call of a user's program through the package's Python API: the conserved
fields are on the GPU, the lattice (or the batch of lattices) exists, and one pass initialises it,
advances it some composite steps and takes the moments, or takes the gradient of the final moments.
The settings (systems, lattice velocities, data) are those of the repository's workloads and tests.

FP32 lattices: the moments come out as doubles, of which a program that computes in float32 keeps
the float32 rounding (they hold no more than that); FP64 lattices' outputs stay doubles.
"""
import math

import torch

from paper_2403_13406_gb300 import autograd, eslbm

G = 9.81
GAMMA = 1.4


def _case(kind, nx, ny=1, steps=1, precision="fp32", mode="entropic", scheme="I", K=0, count=0, lo=0, hi=0):
    return {"kind": kind, "nx": nx, "ny": ny, "steps": steps, "precision": precision, "mode": mode,
            "scheme": scheme, "K": K, "count": count, "lo": lo, "hi": hi}


def listed():
    return [
        # the smallest solve: 1D Burgers on 256 cells to t = 0.5 (convergence tables, interactive use);
        # launches, host work and the chain of stages
        dict(_case("burgers1d", 256, steps=8, precision="fp64"), name="burgers1d_n256_fp64"),
        # the 1D production run: smooth shallow water on 2^20 cells, per-cell entropic omega, FP32 storage
        # shifted by the state at rest
        dict(_case("sw1d", 1 << 20, steps=24), name="sw1d_n1m_fp32"),
        # a dam break: cells at the bore take the root-find's slow branches, the others are at rest
        dict(_case("dambreak", 65536, steps=64), name="sw1d_dambreak_n65536"),
        # the FP64 reference solution that FP32 errors are stated against, on an odd number of cells
        dict(_case("sw1d", 100003, steps=3, precision="fp64"), name="sw1d_n100003_fp64"),
        # FP32 storage with the FP64 certificate of the entropy difference, ragged size
        dict(_case("sw1d", 30001, steps=6, precision="fp32_mixed"), name="sw1d_n30001_mixed"),
        # reverse mode through torch.autograd: data assimilation on one 1D lattice (in FP64: the derivative
        # of the entropic omega divides by the distance from equilibrium, of order dx)
        dict(_case("grad1d", 16384, steps=4, precision="fp64", K=2), name="sw1d_grad_n16384_fp64"),
        # 2D Burgers with noisy data at full size, per-cell entropic omega
        dict(_case("burgers2d", 4096, 4096, steps=4), name="burgers2d_4096"),
        # the 2D convergence study: a Gaussian in FP64, with its entropy totals read back
        dict(_case("gaussian2d", 384, 384, steps=3, precision="fp64"), name="burgers2d_gauss384_fp64"),
        # the largest: 2D Euler, isentropic vortex on 8192^2, fixed omega = 2, larger than any cache
        dict(_case("vortex", 8192, 8192, steps=3, mode="fixed"), name="euler_vortex_8192"),
        # Euler with shocks on a grid whose rows do not start on 16-byte boundaries, the paper's scheme III
        dict(_case("riemann", 1021, 765, steps=10, mode="fixed", scheme="III"), name="euler_riemann_1021x765"),
        # an ensemble of uneven 2D shallow-water lattices advanced together
        dict(_case("batch", 0, 0, steps=4, count=24, lo=256, hi=1024), name="batch_sw2d_24"),
        # its gradient: one optimisation step over an ensemble
        dict(_case("batchgrad", 0, 0, steps=4, K=2, count=6, lo=96, hi=384), name="batch_sw2d_grad_6"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("burgers1d", "sw1d", "sw1d", "dambreak", "grad1d", "burgers2d", "gaussian2d", "vortex", "riemann",
                       "batch", "batchgrad"))
    if kind == "burgers1d":
        n = _log(rng, 128, 20000)  # to t = 1/2 at most, before the shock
        return _case(kind, n, steps=min(rng.randint(4, 24), n // 32), precision=rng.choice(("fp32", "fp64")),
                     mode=rng.choice(("entropic", "entropic", "fixed")))
    if kind == "sw1d":
        precision = rng.choice(("fp32", "fp32", "fp64", "fp32_mixed"))
        if precision == "fp32":
            return _case(kind, _log(rng, 2000, 1 << 20), steps=rng.randint(4, 24))
        return _case(kind, _log(rng, 1000, 100000), steps=rng.randint(1, 4), precision=precision)
    if kind == "dambreak":
        return _case(kind, _log(rng, 4000, 130000), steps=rng.randint(16, 64))
    if kind == "grad1d":
        return _case(kind, _log(rng, 1000, 16000), steps=rng.randint(2, 4), precision="fp64", K=rng.randint(1, 4))
    if kind == "burgers2d":
        return _case(kind, _log(rng, 200, 4096), _log(rng, 200, 4096), steps=rng.randint(2, 4),
                     mode=rng.choice(("entropic", "entropic", "fixed")))
    if kind == "gaussian2d":
        n = _log(rng, 192, 768)  # to t = 1/16 at most
        return _case(kind, n, n + rng.randint(-9, 9), steps=n // 128, precision="fp64")
    if kind == "vortex":  # production grids have rows of whole 16-byte units; the ragged ones are riemann's
        return _case(kind, 4 * _log(rng, 64, 2048), _log(rng, 256, 8192), steps=rng.randint(2, 3), mode="fixed")
    if kind == "riemann":
        return _case(kind, _log(rng, 200, 2000), _log(rng, 200, 2000), steps=rng.randint(4, 10), mode="fixed",
                     scheme=rng.choice(("I", "III")))
    if kind == "batch":
        lo = rng.randint(48, 256)
        return _case(kind, 0, 0, steps=rng.randint(2, 4), count=_log(rng, 4, 24), lo=lo, hi=lo * rng.randint(2, 4))
    lo = rng.randint(48, 128)
    return _case(kind, 0, 0, steps=rng.randint(2, 4), K=2, count=rng.randint(2, 6), lo=lo, hi=lo * rng.randint(2, 3))


# ---------------------------------------------------------------------------
# inputs (on the GPU, from the seed alone)
# ---------------------------------------------------------------------------

def _rand(seed, n, lo, hi):
    """n numbers in [lo, hi) from the seed"""
    return [lo + (hi - lo) * v for v in torch.rand(n, dtype=torch.float64, generator=torch.Generator().manual_seed(seed)).tolist()]


def _axis(n, device, length=1.0):
    return torch.arange(n, dtype=torch.float64, device=device) * (length / n)


def _sizes(case):
    """uneven (nx, ny) of a batch: those of the case, whatever the seed of the data"""
    g = torch.Generator().manual_seed(7 + case["count"])
    return [tuple(v) for v in torch.randint(case["lo"], case["hi"] + 1, (case["count"], 2), generator=g).tolist()]


def _sw_fourier(nx, ny, seed, device):
    """depth 1 + 0.05 times eight seeded Fourier modes, at rest"""
    r = _rand(seed, 32, 0.0, 1.0)
    x, y = _axis(nx, device)[None, :], _axis(ny, device)[:, None]
    h = torch.ones((ny, nx), dtype=torch.float64, device=device)
    amp = [2.0 * v - 1.0 for v in r[:8]]
    norm = sum(abs(a) for a in amp)
    for m in range(8):
        kx, ky = int(r[8 + m] * 9) - 4, int(r[16 + m] * 9) - 4
        if kx == ky == 0:
            kx = 1
        h += 0.05 * amp[m] / norm * torch.cos(2 * math.pi * (kx * x + ky * y) + 2 * math.pi * r[24 + m])
    return torch.stack([h, torch.zeros_like(h), torch.zeros_like(h)])


def _fields(case, seed, device):
    """initial conserved fields of a single lattice: (M, [ny,] nx) doubles"""
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    r = _rand(seed, 16, 0.0, 1.0)
    if kind == "burgers1d":
        return (0.5 + (0.2 + 0.05 * r[0]) * torch.sin(2 * math.pi * (_axis(nx, device) + r[1])))[None]
    if kind in ("sw1d", "grad1d"):
        h = 1.0 + (0.08 + 0.04 * r[0]) * torch.sin(2 * math.pi * (_axis(nx, device) + r[1]))
        return torch.stack([h, torch.zeros_like(h)])
    if kind == "dambreak":
        x = _axis(nx, device)
        h = torch.where(x < 0.4 + 0.2 * r[0], 1.8 + 0.4 * r[1], 1.0).to(torch.float64)
        return torch.stack([h, torch.zeros_like(h)])
    if kind == "burgers2d":
        x, y = _axis(nx, device)[None, :], _axis(ny, device)[:, None]
        u = 0.5 + 0.25 * torch.sin(2 * math.pi * (x + r[0])) * torch.sin(2 * math.pi * (y + r[1]))
        g = torch.Generator(device=device).manual_seed(seed)
        return (u + 1e-3 * torch.randn((ny, nx), dtype=torch.float64, device=device, generator=g))[None]
    if kind == "gaussian2d":
        x, y = _axis(nx, device)[None, :], _axis(ny, device)[:, None]
        return torch.exp(-(80.0 + 20.0 * r[2]) * ((x - 0.4 - 0.2 * r[0]) ** 2 + (y - 0.4 - 0.2 * r[1]) ** 2))[None]
    if kind == "vortex":
        x, y = _axis(nx, device, 10.0)[None, :] - 4.5 - r[0], _axis(ny, device, 10.0)[:, None] - 4.5 - r[1]
        s = 4.5 + r[2]
        e = torch.exp(0.5 * (1.0 - x * x - y * y))
        rho = (1.0 - (GAMMA - 1.0) * s * s / (8 * GAMMA * math.pi ** 2) * e * e) ** (1.0 / (GAMMA - 1.0))
        u, v = 1.0 - s / (2 * math.pi) * e * y, 1.0 + s / (2 * math.pi) * e * x
        return torch.stack([rho, rho * u, rho * v, rho ** GAMMA / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])
    if kind == "riemann":
        q = _rand(seed + 1, 18, 0.0, 1.0)
        x, y = _axis(nx, device)[None, :], _axis(ny, device)[:, None]
        out = torch.zeros((4, ny, nx), dtype=torch.float64, device=device)
        for i in range(4):
            rho, p, u, v = 0.5 + q[4 * i], 0.5 + q[4 * i + 1], q[4 * i + 2] - 0.5, q[4 * i + 3] - 0.5
            here = ((x >= 0.3 + 0.4 * q[16]) == bool(i & 1)) & ((y >= 0.3 + 0.4 * q[17]) == bool(i & 2))
            for m, w in enumerate((rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v))):
                out[m] += here * w
        return out
    raise ValueError(kind)


#: settings of the lattices, as the repository's workloads and tests have them
SETTINGS = {
    "burgers1d": dict(dim=1, system="burgers", V=1.5),
    "sw1d": dict(dim=1, system="sw", V=4.0, g=G),
    "grad1d": dict(dim=1, system="sw", V=4.0, g=G),
    "dambreak": dict(dim=1, system="sw", V=6.0 * math.sqrt(G), g=G),
    "burgers2d": dict(dim=2, system="burgers", V=3.0),
    "gaussian2d": dict(dim=2, system="burgers", V=3.0, c=(1.0, 0.6)),
    "vortex": dict(dim=2, system="euler", V=8.0, gamma=GAMMA),
    "riemann": dict(dim=2, system="euler", V=8.0, gamma=GAMMA, omega=1.98),
    "batch": dict(dim=2, system="sw", V=8.0, g=G),
    "batchgrad": dict(dim=2, system="sw", V=8.0, g=G),
}

_streams = []


def _stream():
    """the program's stream (CUDA graphs need one that is not the default)"""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def _config(case):
    kw = dict(SETTINGS[case["kind"]])
    if case["kind"] == "sw1d" and case["precision"] != "fp64":
        kw["u_ref"] = (1.0, 0.0)  # the depth at rest: FP32 storage of the deviations from it
    if case["kind"] in ("batch", "batchgrad"):
        kw["u_ref"] = (1.0, 0.0, 0.0)
    return eslbm.make_config(kw.pop("dim"), kw.pop("system"), max(1, case["nx"]), max(1, case["ny"]), precision=case["precision"],
                             omega_mode=case["mode"], scheme=case["scheme"], **kw)


def _batch_fields(case, seed, device):
    return [_sw_fourier(nx, ny, 1000 * seed + i, device) for i, (nx, ny) in enumerate(_sizes(case))]


def _cotangents(fields, targets):
    """dJ/du_T of the misfit in depth between two sets of fields"""
    out = []
    for u, t in zip(fields, targets):
        lam = torch.zeros_like(u)
        lam[0] = 2.0 * (u[0] - t[0])
        out.append(lam)
    return out


def prepare(case, seed):
    stream = _stream()
    cfg = _config(case)
    with torch.cuda.stream(stream):
        s = {"case": case, "stream": stream}
        if case["kind"] in ("batch", "batchgrad"):
            b = s["batch"] = eslbm.Batch(cfg, _sizes(case), stream=stream)
            b.use_graph(True)
            fields = _batch_fields(case, seed, "cuda")
            s["u0"] = b.pack(fields)
            if case["kind"] == "batchgrad":
                s["lam"] = b.pack(_cotangents(fields, _batch_fields(case, seed + 4000, "cuda")))
        else:
            sim = s["sim"] = eslbm.Simulation(cfg, stream=stream)
            sim.use_graph(True)
            s["u0"] = _fields(case, seed, "cuda")
            if case["kind"] == "grad1d":
                s["lam"] = _cotangents([s["u0"]], [_fields(case, seed + 4000, "cuda")])[0]
                s["u0"].requires_grad_(True)
    stream.synchronize()
    return s


def run(state):
    case = state["case"]
    fp32 = case["precision"] != "fp64"
    with torch.cuda.stream(state["stream"]):
        if case["kind"] == "batch":
            b = state["batch"]
            b.init_equilibrium(state["u0"])
            b.step(case["steps"])
            return b.moments_flat().float()
        if case["kind"] == "batchgrad":
            return state["batch"].gradient(state["u0"], state["lam"], case["steps"], case["K"]).float()
        sim = state["sim"]
        if case["kind"] == "grad1d":
            uT = autograd.evolve(state["u0"], sim, case["steps"], case["K"])
            (du0,) = torch.autograd.grad(uT, state["u0"], state["lam"])
            return {"uT": uT.detach(), "du0": du0}
        sim.init_equilibrium(state["u0"])
        sim.step(case["steps"])
        u = sim.moments()
        if case["kind"] == "gaussian2d":
            return {"u": u, "totals": sim.totals(host=False)}
        return u.float() if fp32 else u


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _cells(case):
    return sum(nx * ny for nx, ny in _sizes(case)) if case["count"] else case["nx"] * case["ny"]


def _dim_m(case):
    dim, system = SETTINGS[case["kind"]]["dim"], SETTINGS[case["kind"]]["system"]
    return dim, {"burgers": 1, "sw": dim + 1, "euler": 4}[system]


def work(case):
    """bytes: the initial fields (doubles) read once and the outputs written once.  flops: per cell and
    relaxation the moments, the equilibrium, the deviations and the update, the entropic omega as
    twice that again (an expansion of the entropy about the equilibrium), a reverse sweep as two more."""
    dim, M = _dim_m(case)
    q = 2 * dim
    stages = {"I": 18, "III": 27}[case["scheme"]]
    cells, out = _cells(case), 8 if case["precision"] == "fp64" else 4
    relax = q * M * 6 + 6 * M
    if case["mode"] == "entropic":
        relax *= 3
    n_in, n_out, sweeps = 1, 1, 1
    if case["kind"] in ("grad1d", "batchgrad"):
        n_in, sweeps = 2, 3
        n_out = 2 if case["kind"] == "grad1d" else 1
    return {"bytes": cells * M * (8 * n_in + out * n_out), "flops": cells * case["steps"] * stages * relax * sweeps}


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch's own operations
# ---------------------------------------------------------------------------

def _shifts(scheme):
    """(transport, projection) before each relaxation of one step, and the transport after the last"""
    ops = []
    pend = 0
    for q4, reps in ((1, 4), (-2, 1), (1, 4)):
        for _ in range(reps):
            ops.append((pend + q4, False))
            ops.append((2 * q4, False))
            pend = q4
            if scheme == "III":
                ops.append((pend, True))
                pend = 0
    return ops, pend


class _Model:
    """f: (q, M, cells); velocities +x, (+y,) -x, (-y); the lattices' cells one after the other"""

    def __init__(self, case, shapes):
        kw = SETTINGS[case["kind"]]
        self.system, self.dim, self.V = kw["system"], kw["dim"], kw["V"]
        self.q = 2 * self.dim
        self.c = kw.get("c", (1.0, 1.0))
        self.omega, self.entropic = kw.get("omega", 2.0), case["mode"] == "entropic"
        self.shapes = [tuple(v) for v in shapes]
        self.axes = [k % self.dim for k in range(self.q)]
        self.signs = [1.0 if k < self.dim else -1.0 for k in range(self.q)]

    def flux(self, j, u):
        if self.system == "burgers":
            return (0.5 * self.c[j]) * u * u
        if self.system == "sw":
            v = u[1 + j] / u[0]
            out = [u[1 + i] * v for i in range(self.dim)]
            out[j] = out[j] + 0.5 * G * u[0] * u[0]
            return torch.stack([u[1 + j]] + out)
        vj = u[1 + j] / u[0]
        p = (GAMMA - 1.0) * (u[3] - 0.5 * (u[1] * u[1] + u[2] * u[2]) / u[0])
        out = [u[1 + j], u[1] * vj, u[2] * vj, (u[3] + p) * vj]
        out[1 + j] = out[1 + j] + p
        return torch.stack(out)

    def equilibrium(self, u):
        phi = [self.flux(j, u) / (2.0 * self.V) for j in range(self.dim)]
        return torch.stack([u / self.q + sg * phi[j] for j, sg in zip(self.axes, self.signs)])

    def entropy_of(self, u, d):
        """t -> the sum over the populations of the Bregman divergence of the kinetic entropy for the
        increments t d, and its derivative in t; and the largest t to look at (3, or less where a
        population leaves the domain)"""
        sg = torch.tensor(self.signs, dtype=u.dtype, device=u.device)[:, None]
        if self.system == "burgers":
            c = sg * torch.tensor([self.c[j] for j in self.axes], dtype=u.dtype, device=u.device)[:, None]
            D = 1.0 / self.q + c * u[0] / (2.0 * self.V)  # second derivative of the dual entropy
            x1, a = (c / self.V) * d[:, 0] / (D * D), d[:, 0] * d[:, 0] / D

            def scalar(t):
                s = torch.sqrt(1.0 + t * x1)
                return (a * (1.0 + 2.0 * s) / ((1.0 + s) * (1.0 + s))).sum(0) * (2.0 / 3.0) * t * t, (a / (1.0 + s)).sum(0) * 2.0 * t

            return scalar, torch.where(x1 < 0, -1.0 / x1, 3.0).amin(0).clamp(max=3.0)
        # shallow water: s_k(f) = max over p of g V f_1^2 / (nu + sg p) - p^2 f_1 / 2 + p f_d, plus f_t^2 / (2 f_1)
        # across the axis; with f_1 = equilibrium (1 + eta), p = v - sg c beta it is f_1 c^2 times
        #   K (eta + beta)^2 / (1 - beta) - R beta - (1 + eta) beta^2 / 2
        v = torch.stack([u[1 + j] / u[0] for j in self.axes])
        dd = torch.stack([d[k, 1 + j] for k, j in enumerate(self.axes)])
        c = 2.0 * self.V / self.q + sg * v
        f1 = u[0] * c / (2.0 * self.V)
        K = 0.5 * G * u[0] / (c * c)
        e1, R1, w = d[:, 0] / f1, sg * (dd - v * d[:, 0]) / (f1 * c), f1 * c * c
        z = 0.0
        if self.dim == 2:
            vt = torch.stack([u[2 - j] / u[0] for j in self.axes])
            z = 0.5 * (torch.stack([d[k, 2 - j] for k, j in enumerate(self.axes)]) - vt * d[:, 0]) ** 2 / f1

        def water(t):
            eta, R = t * e1, t * R1
            beta = (2.0 * K * eta - R) / (1.0 - 2.0 * K)
            for _ in range(6):
                r = 1.0 / (1.0 - beta)
                g = K * (eta + beta) * (2.0 + eta - beta) * r * r - (1.0 + eta) * beta - R
                beta = beta - g / ((1.0 + eta) * (2.0 * K * (1.0 + eta) * r ** 3 - 1.0))
            s = (eta + beta) / (1.0 - beta)
            b = w * (K * (eta + beta) * s - R * beta - 0.5 * (1.0 + eta) * beta * beta) + z * t * t / (1.0 + eta)
            db = w * ((2.0 * K * s - 0.5 * beta * beta) * e1 - beta * R1) + z * t * (2.0 + eta) / (1.0 + eta) ** 2
            return b.sum(0), db.sum(0)

        return water, torch.where(e1 < 0, -1.0 / e1, 3.0).amin(0).clamp(max=3.0)

    def relax(self, f, project=False):
        u = f.sum(0)
        if not self.entropic or project:
            return f.lerp_(self.equilibrium(u), 1.0 if project else self.omega)
        d = self.equilibrium(u) - f
        with torch.no_grad():
            B, most = self.entropy_of(u.detach(), d.detach())
            t = torch.ones_like(u[0])
            e0 = B(-t)[0]
            for _ in range(20):  # the imbalance is convex in t: from the right of the root Newton stays there
                b, db = B(t)
                move = torch.where(e0 > 0, (b - e0) / db, 0.0)
                t = torch.minimum(t - move, most)
                if float(torch.where(t < most, move, 0.0).abs().max()) < 1e-13:
                    break
            t = torch.where(t < most, t, 0.0)  # no root inside the domain: the projection
        if f.requires_grad:  # one step more, differentiated: the implicit function theorem
            B, _ = self.entropy_of(u, d)
            b, db = B(t)
            t = t - torch.where(e0 > 0, (b - B(-torch.ones_like(t))[0]) / db.detach(), 0.0)
        return f + (1.0 + t) * d

    def transport(self, f, s):
        """population k moves s cells along its velocity; a lattice's cells are (ny, nx) or (nx,)"""
        out, at = [], 0
        for shape in self.shapes:
            n = math.prod(shape)
            part = f[:, :, at:at + n].reshape(f.shape[:2] + shape)
            out.append(torch.stack([torch.roll(part[k], int(self.signs[k]) * s, dims=-1 - self.axes[k])
                                    for k in range(self.q)]).flatten(2))
            at += n
        return out[0] if len(out) == 1 else torch.cat(out, 2)


def _exact_stages(case):
    """(transport, projection) of all relaxations of the case, and the transport after them"""
    ops, trail = _shifts(case["scheme"])
    out, pend = [], 0
    for _ in range(case["steps"]):
        for i, (s, p) in enumerate(ops):
            out.append((s + (pend if i == 0 else 0), p))
        pend = trail
    return out, pend


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    many = case["count"] > 0
    fields = _batch_fields(case, seed, dev) if many else [_fields(case, seed, dev)]
    shapes = [tuple(u.shape[1:]) for u in fields]
    model = _Model(case, shapes)
    pack = lambda parts: torch.cat([p.reshape(p.shape[0], -1) for p in parts], 1)

    def unpack(u):  # one lattice after the other, as the batch lays them out
        parts = torch.split(u, [math.prod(s) for s in shapes], 1)
        return torch.cat([p.reshape(-1) for p in parts]) if many else u.reshape(u.shape[:1] + shapes[0])

    stages, trail = _exact_stages(case)
    u0 = pack(fields)
    f = model.equilibrium(u0)
    if case["kind"] not in ("grad1d", "batchgrad"):
        del fields, u0
        for s, project in stages:
            f = model.relax(model.transport(f, s), project)
        u = unpack(model.transport(f, trail).sum(0))
        return {"u": u, "totals": None} if case["kind"] == "gaussian2d" else u
    inputs = []
    for s, project in stages:
        inputs.append(model.transport(f, s))
        f = model.relax(inputs[-1], project)
    uT = model.transport(f, trail).sum(0)
    targets = _batch_fields(case, seed + 4000, dev) if many else [_fields(case, seed + 4000, dev)]
    lam = pack(_cotangents(fields, targets))
    g = model.transport(lam.expand((model.q,) + lam.shape), -trail)
    for (s, project), f in zip(reversed(stages), reversed(inputs)):
        f = f.requires_grad_(True)
        with torch.enable_grad():
            (g,) = torch.autograd.grad(model.relax(f, project), f, g)
        g = model.transport(g, -s)
        f.requires_grad_(False)
    u0.requires_grad_(True)
    with torch.enable_grad():
        (du0,) = torch.autograd.grad(model.equilibrium(u0), u0, g)
    return unpack(du0) if many else {"uT": unpack(uT), "du0": unpack(du0)}
