"""Performance cases of the MG-GLAM field solver: what its users have it do.

Each case is one call, or one short chain of calls, of the public entry points
(paper_2110_00328_gb300.binding and .autograd), on inputs made on the GPU from a
seed: particles on a lattice displaced by a Zel'dovich field, and lognormal
densities, with the statistics of paper_2110_00328_gb300/inputs.py.  Every
solve starts from the background field, as a first time step or an emulator's
does, except the particle-mesh step's, which starts from the previous field.

The coupled-quintessence equation leaves the mean of its field undetermined (its
mass is 1e-8 of the mesh's), so the case returns what a program takes from it:
the forces, and the field about its mean.
"""
import math
import random

import torch

from paper_2110_00328_gb300 import autograd, binding

C_H0 = 299792.458 / 100.0  # c/H0 in Mpc/h
OM, OL = 0.3, 0.7
A_STAR = 0.5
# lambda and phibar(a = 1) of the coupled-quintessence background (alpha = 0.1, beta = -0.05, Om = 0.3, h = 0.6774)
CQ_LAM, CQ_PHIBAR, CQ_ALPHA, CQ_BETA = 1.440377, 0.779528, 0.1, -0.05
# sides whose multigrid hierarchy reaches 4, 6, 10 or 14 cells, up to those the largest meshes use
SIDES = [32, 40, 48, 56, 64, 80, 96, 112, 128, 160, 192, 224, 256, 320]


def listed():
    return [
        # the small parity solve of the tests: a parameter scan's or a coarse simulation's mesh, bound by latency
        dict(name="solve_fr_32", kind="solve", model="fr", n=1, N=32, box=64.0, fr0=1e-5, sigma=1.0, tol=1e-10,
             nu1=2, nu2=2, sweeps=16, fp64=False),
        # the benchmark's solve: one time step's field equation of an F6 run, strongly screened
        dict(name="solve_fr_256", kind="solve", model="fr", n=1, N=256, box=256.0, fr0=1e-6, sigma=1.5, tol=1e-8,
             nu1=2, nu2=1, sweeps=4, fp64=False),
        # the symmetron on a mesh that is no power of two
        dict(name="solve_sym_192", kind="solve", model="sym", n=1, N=192, box=192.0, range=1.0, sigma=1.5, tol=1e-8,
             nu1=2, nu2=2, sweeps=16, fp64=False),
        # coupled quintessence: field and forces
        dict(name="forces_cq_128", kind="solve", model="cq", n=1, N=128, box=128.0, sigma=1.5, tol=1e-10, nu1=2,
             nu2=1, sweeps=4, fp64=False, M=64),
        # the plain-FP64 solve: validation runs and whoever wants no mixed precision
        dict(name="solve_fr_fp64_96", kind="solve", model="fr", n=1, N=96, box=96.0, fr0=1e-5, sigma=1.0, tol=1e-10,
             nu1=2, nu2=2, sweeps=16, fp64=True),
        # the single-step entry points, composed to a two-grid cycle by a caller with a cycle of their own
        dict(name="twogrid_fr_128", kind="twogrid", model="fr", n=1, N=128, box=128.0, fr0=1e-5, sigma=1.0),
        # density of as many particles as cells (the benchmark's step)
        dict(name="deposit_256", kind="deposit", N=256, M=256, sigma=1.5),
        # fifth force on as many particles as cells (the benchmark's step)
        dict(name="gather_fr_256", kind="gather", model="fr", n=1, N=256, M=256, box=256.0, fr0=1e-6, sigma=1.5),
        # gradient of a loss through the solve, forward and backward: inference and emulator training
        dict(name="gradient_fr_512", kind="gradient", model="fr", n=1, N=512, box=512.0, fr0=1e-5, sigma=1.5,
             tol=1e-10),
        # an emulator's parameter grid: many small solves of both models at once
        dict(name="batch_12", kind="batch", count=12, mix=4, tol=1e-8),
        # Newtonian gravity
        dict(name="poisson_256", kind="poisson", N=256, sigma=1.5),
        # one whole time step of a modified-gravity simulation, the mesh twice as fine as the particles
        dict(name="pm_fr_256", kind="pm", model="fr", n=1, N=256, M=128, box=256.0, fr0=1e-6, sigma=1.5, tol=1e-8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _model(rng, c, models):
    c["model"] = rng.choice(models)
    c["n"] = rng.choice([0, 1, 1, 1, 2]) if c["model"] == "fr" else 1
    c["box"] = c["N"] * rng.choice([1.0, 1.0, 2.0])
    if c["model"] == "fr":
        c["fr0"] = _log(rng, 1e-6, 2e-5)
    elif c["model"] == "sym":
        c["range"] = _log(rng, 0.5, 3.0) * c["box"] / c["N"]
    return c


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "twogrid", "deposit", "gather", "gradient", "batch", "poisson", "pm"])
    c = dict(kind=kind, sigma=round(rng.uniform(0.8, 1.8), 3))
    if kind == "solve":
        c["fp64"] = rng.random() < 0.25
        c["N"] = rng.choice(SIDES[:10] if c["fp64"] else SIDES)
        _model(rng, c, ["fr", "fr", "sym", "cq"])
        c["tol"] = 1e-10 if c["model"] == "cq" else rng.choice([1e-9, 1e-10] if c["N"] < 128 else [1e-8, 1e-9, 1e-10])
        c["nu1"], c["nu2"], c["sweeps"] = rng.choice([(2, 2, 16), (2, 1, 4)])
        if c["model"] == "cq":
            c["N"] = rng.choice([32, 48, 64, 96, 128, 192] if not c["fp64"] else [32, 48, 64, 96])
            c["box"] = float(c["N"])
            c["M"] = rng.randint(20, c["N"])
    elif kind == "twogrid":
        c["N"] = 4 * rng.randint(6, 48)
        _model(rng, c, ["fr", "fr", "sym", "cq"])
    elif kind == "deposit":
        c["N"] = 2 * rng.randint(16, 192)
        c["M"] = round(_log(rng, 24, 256))
    elif kind == "gather":
        c["N"] = rng.choice(SIDES)
        c["M"] = round(_log(rng, 24, 256))
        _model(rng, c, ["fr", "sym", "cq"])
    elif kind == "gradient":
        c["N"] = rng.choice([32, 48, 64, 96, 128, 160, 192, 256])
        _model(rng, c, ["fr", "fr", "sym"])
        c["tol"] = 1e-10
    elif kind == "batch":
        c["count"], c["mix"], c["tol"] = rng.randint(3, 16), rng.randrange(1 << 20), 1e-8
    elif kind == "poisson":
        c["N"] = rng.choice([16, 32, 64, 128, 256, 512])
    else:
        c["N"] = rng.choice([32, 64, 128, 256])
        c["M"] = rng.randint(c["N"] // 2, c["N"]) if c["N"] < 256 else rng.choice([128, 160, 256])
        _model(rng, c, ["fr", "sym", "lcdm"])
        c["tol"] = 1e-9
    return c


def _batch_members(c):
    """(side, parameters) of a batch's solves: sides and parameters of the benchmark's batch."""
    r = random.Random(c["mix"])
    out = []
    for _ in range(c["count"]):
        N = r.choice([64, 64, 96, 96, 128])
        d = dict(N=N, box=float(N), n=1, sigma=r.uniform(0.8, 1.8), nu1=2, nu2=2, sweeps=16, tol=c["tol"])
        if r.random() < 0.5:
            d.update(model="fr", fr0=_log(r, 1e-7, 1e-4))
        else:
            d.update(model="sym", range=_log(r, 0.5, 3.0))
        out.append(d)
    return out


def _params(c, fp64=False):
    kw = dict(box=c["box"], precision=binding.FP64 if fp64 else binding.MIXED, max_cycles=80, nu1=c.get("nu1", 2),
              nu2=c.get("nu2", 2), coarse_sweeps=c.get("sweeps", 16))
    if c["model"] in ("fr", "lcdm"):
        return binding.Params(model=binding.FR, n=c["n"], fR0_abs=c.get("fr0", 1e-5), **kw)
    if c["model"] == "sym":
        return binding.Params(model=binding.SYMMETRON, a_star=A_STAR, beta_star=1.0, xi=c["range"] / C_H0, **kw)
    return binding.Params(model=binding.CQ, alpha=CQ_ALPHA, beta=CQ_BETA, lam=CQ_LAM, phibar=CQ_PHIBAR, **kw)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _k(N):
    kx = 2.0 * math.pi * torch.fft.fftfreq(N, device="cuda", dtype=torch.float64)
    kz = 2.0 * math.pi * torch.fft.rfftfreq(N, device="cuda", dtype=torch.float64)
    return kx[:, None, None], kx[None, :, None], kz[None, None, :]


def _gaussian_k(N, seed, slope, sharp):
    """rfftn of a Gaussian field with P ~ k^slope and a Gaussian cut at half the Nyquist wavenumber, or a sharp one at it."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f = torch.fft.rfftn(torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64))
    kx, ky, kz = _k(N)
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    f *= k2 ** (0.25 * slope)
    f *= (k2 <= math.pi ** 2).double() if sharp else torch.exp(-0.5 * k2 / (0.5 * math.pi) ** 2)
    f[0, 0, 0] = 0.0
    return f, k2


def _density(N, sigma, seed):
    """Lognormal density of mean 1, float32."""
    f, _ = _gaussian_k(N, seed, -1.5, False)
    g = torch.fft.irfftn(f, s=(N, N, N))
    g *= sigma / g.std()
    rho = torch.exp(g - 0.5 * sigma * sigma)
    return (rho / rho.mean()).float().contiguous()


def _particles(N, M, sigma, seed, margin=0.0):
    """M^3 Zel'dovich particles in cell units of an N^3 mesh (float32) and their displacements."""
    f, k2 = _gaussian_k(M, seed, -2.0, True)
    f *= sigma / torch.fft.irfftn(f, s=(M, M, M)).std()
    f /= k2
    q = torch.arange(M, device="cuda", dtype=torch.float64) + 0.5
    base = (q[:, None, None], q[None, :, None], q[None, None, :])
    psi = torch.stack([torch.fft.irfftn(1j * k * f, s=(M, M, M)) for k in _k(M)], dim=-1)
    pos = torch.stack([(base[d] + psi[..., d]) * (N / M) for d in range(3)], dim=-1).remainder_(float(N))
    if margin:
        pos.clamp_(margin, N - margin)
    pos = pos.reshape(-1, 3).float()
    pos[pos >= N] = 0.0
    return pos.contiguous(), (psi.reshape(-1, 3) * (N / M)).float().contiguous()


def _field(c, seed):
    """A field of the size and smoothness of a solution: below the background in dense regions."""
    N = c["N"]
    rho = _density(N, c["sigma"], seed).double()
    smooth = torch.nn.functional.avg_pool3d(torch.nn.functional.pad(rho[None, None], (1,) * 6, mode="circular"), 3, 1)[0, 0]
    if c["model"] == "cq":
        return (1e-3 * (smooth - 1.0)).contiguous()
    m = _Model(c)
    return (m.ubar / (1.0 + 0.2 * smooth)).contiguous()


NAN = float("nan")


def _background(N):
    return torch.full((N, N, N), NAN, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    c = dict(case)
    s = dict(c=c, kind=c["kind"])
    N = c.get("N")
    mark = torch.tensor([NAN], dtype=torch.float64).pin_memory()  # "start from the background"
    if c["kind"] == "solve":
        s.update(prm=_params(c, c["fp64"]), rho=_density(N, c["sigma"], seed), field=_background(N), mark=mark)
        if c["model"] == "cq":
            s["pos"] = _particles(N, c["M"], c["sigma"], seed + 1)[0]
    elif c["kind"] == "twogrid":
        rho = _density(N, c["sigma"], seed).double()
        s.update(prm=_params(c), rho=(rho / rho.mean()).contiguous(), u0=_field(c, seed + 1))
        s["rhoH"] = binding.restrict(s["rho"])
    elif c["kind"] == "deposit":
        s.update(pos=_particles(N, c["M"], c["sigma"], seed)[0],
                 rho=torch.empty((N, N, N), dtype=torch.float32, device="cuda"))
    elif c["kind"] == "gather":
        s.update(prm=_params(c), field=_field(c, seed + 1), pos=_particles(N, c["M"], c["sigma"], seed)[0])
        s["force"] = torch.empty_like(s["pos"])
    elif c["kind"] == "gradient":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        s.update(prm=_params(c), rho=_density(N, c["sigma"], seed),
                 theta=torch.tensor(math.log(c.get("fr0", 1e-5)), dtype=torch.float64),
                 g=torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64))
    elif c["kind"] == "batch":
        mem = _batch_members(c)
        s.update(prm=[_params(m) for m in mem], mark=mark, fields=[_background(m["N"]) for m in mem],
                 rhos=[_density(m["N"], m["sigma"], seed + 7 * i) for i, m in enumerate(mem)])
    elif c["kind"] == "poisson":
        s.update(rho=_density(N, c["sigma"], seed), phi=torch.empty((N, N, N), dtype=torch.float32, device="cuda"))
    else:
        # no particle starts at a face of the box: where it lands, 0 and N are the same place on its last bit
        pos, psi = _particles(N, c["M"], c["sigma"], seed, margin=0.3)
        a, da = 0.9, 0.01
        s.update(prm=_params(dict(c, nu2=1, sweeps=4)), a=a, da=da, pos0=pos, mom0=psi * (a * a * _E(a)),
                 pos=pos.clone(), mom=torch.empty_like(pos), field0=None, field=None)
        s["rho"], s["psi"] = (torch.empty((N, N, N), dtype=torch.float32, device="cuda") for _ in range(2))
        if c["model"] != "lcdm":  # the previous step's field
            s["field0"], s["field"] = _background(N), _background(N)
            binding.deposit_cic((pos - psi * (da / a)).remainder(float(N)).contiguous(), N, s["rho"])
            binding.solve_scalar(s["prm"], a - da, s["rho"], s["field0"], c["tol"])
    return s


def _E(a):
    return math.sqrt(OM / a ** 3 + OL)


def run(s):
    c, kind = s["c"], s["kind"]
    if kind == "solve":
        field = s["field"]
        field.view(-1)[:1].copy_(s["mark"], non_blocking=True)
        binding.solve_scalar(s["prm"], 1.0, s["rho"], field, c["tol"])
        if c["model"] != "cq":
            return {"field": field}
        return {"field": field - field.mean(), "force": binding.gather_force(s["prm"], 1.0, field, s["pos"])}
    if kind == "twogrid":
        prm, rho, rhoH, u = s["prm"], s["rho"], s["rhoH"], s["u0"].clone()
        binding.smooth(prm, 1.0, u, rho, sweeps=2)
        d, _ = binding.residual(prm, 1.0, u, rho)
        uH = binding.restrict(u)
        RuH, dH = uH.clone(), binding.restrict(d)
        NH, _ = binding.residual(prm, 1.0, uH, rhoH, h=2.0)
        binding.smooth(prm, 1.0, uH, rhoH, S=NH - dH, sweeps=2, h=2.0)
        binding.prolong_correct(prm, uH, RuH, u)
        binding.smooth(prm, 1.0, u, rho, sweeps=2)
        d, _ = binding.residual(prm, 1.0, u, rho)
        return {"u": u, "uH": uH, "d": d}
    if kind == "deposit":
        return binding.deposit_cic(s["pos"], c["N"], s["rho"])
    if kind == "gather":
        return binding.gather_force(s["prm"], 1.0, s["field"], s["pos"], 1.0, s["force"])
    if kind == "gradient":
        rho, theta = s["rho"].detach().requires_grad_(True), s["theta"].detach().requires_grad_(True)
        u = autograd.solve(rho, theta, s["prm"], 1.0, c["tol"])
        u.backward(s["g"])
        return {"field": u.detach(), "grad_rho": rho.grad, "grad_log_fr0": theta.grad}
    if kind == "batch":
        for f in s["fields"]:
            f.view(-1)[:1].copy_(s["mark"], non_blocking=True)
        binding.solve_batch(s["prm"], [1.0] * c["count"], s["rhos"], s["fields"], c["tol"])
        return s["fields"]
    if kind == "poisson":
        return binding.poisson_fft(s["rho"], 1.5 * OM, s["phi"])
    # every pass is the same step of a simulation: it starts from the same particles and field
    s["pos"].copy_(s["pos0"])
    s["mom"].copy_(s["mom0"])
    if s["field"] is not None:
        s["field"].copy_(s["field0"])
    binding.pm_step(s["prm"], s["a"], s["da"], s["pos"], s["mom"], s["rho"], s["psi"], field=s["field"], tol=c["tol"])
    out = {"pos": s["pos"], "mom": s["mom"]}
    return out if s["field"] is None else dict(out, field=s["field"])


def work(case):
    """Inputs read and outputs written once; operations of one relaxation and one residual of every cell (solves),
    of the 8 or 32 cells a particle meets, and of one real transform each way (5/2 N log2 N)."""
    c = dict(case)
    if c["kind"] == "batch":
        n3 = sum(m["N"] ** 3 for m in _batch_members(c))
        return {"bytes": 12.0 * n3, "flops": 60.0 * n3}
    n3, p3 = float(c["N"]) ** 3, float(c.get("M", 0)) ** 3
    fft = 5.0 * n3 * 3 * math.log2(c["N"])
    if c["kind"] == "solve":
        return {"bytes": 12.0 * n3 + (8.0 * n3 + 24.0 * p3 if c["model"] == "cq" else 0.0), "flops": 60.0 * n3 + 100.0 * p3}
    if c["kind"] == "twogrid":
        return {"bytes": (24.0 + 8.0 / 8) * n3 + 8.0 * n3, "flops": 250.0 * n3}
    if c["kind"] == "deposit":
        return {"bytes": 12.0 * p3 + 4.0 * n3, "flops": 30.0 * p3}
    if c["kind"] == "gather":
        return {"bytes": 24.0 * p3 + 8.0 * n3, "flops": 100.0 * p3}
    if c["kind"] == "gradient":
        return {"bytes": (4.0 + 8.0) * n3 + (8.0 + 4.0) * n3, "flops": 120.0 * n3}
    if c["kind"] == "poisson":
        return {"bytes": 8.0 * n3, "flops": fft}
    scalar = c["model"] != "lcdm"
    return {"bytes": 48.0 * p3 + (16.0 * n3 if scalar else 0.0), "flops": 130.0 * p3 + fft + (60.0 * n3 if scalar else 0.0)}


# ---------------------------------------------------------------------------
# The same results in 64 bits, by other methods (Newton's method on the whole
# mesh, linear systems by conjugate gradients), without the package's code
# ---------------------------------------------------------------------------

class _Model:
    """Constants of the discrete equation N(u) = 0 at scale factor a (cell size 1)."""

    def __init__(self, c, a=1.0):
        self.kind, self.n = c["model"], c["n"]
        self.c2 = (c["N"] / c["box"] * C_H0) ** 2
        self.om_a = OM / a
        if self.kind == "fr":
            R = lambda x: 3.0 * (OM / x ** 3 + 4.0 * OL)
            self.ubar = (c["fr0"] * (R(1.0) / R(a)) ** (self.n + 1)) ** (1.0 / (self.n + 1))
            self.K0 = R(a) * a * a / 3.0
            self.K = self.K0 * self.ubar
        elif self.kind == "sym":
            self.xi = c["range"] / C_H0
            self.r3 = (A_STAR / a) ** 3
            self.ubar = math.sqrt(1.0 - self.r3)
            self.ms = a * a / (2.0 * self.xi ** 2)
        else:
            self.ubar = 0.0
            self.src = 3.0 * CQ_BETA * OM * math.exp(CQ_BETA * CQ_PHIBAR) / a
            self.pot = CQ_ALPHA * CQ_LAM ** 2 * a * a

    def w(self, u):
        return u ** (self.n + 1) if self.kind == "fr" else u

    def N(self, u, rho, h=1.0):
        k = self.c2 / (h * h)
        if self.kind == "fr":
            return -k * _lap(self.w(u)) + self.om_a * (rho - 1.0) + self.K0 - self.K / u
        if self.kind == "sym":
            return k * _lap(u) - self.ms * ((rho * self.r3 - 1.0) * u + u ** 3)
        x = CQ_PHIBAR + u / self.c2
        return _lap(u) / (h * h) - self.src * (rho - 1.0) + self.pot * (x ** (-1.0 - CQ_ALPHA) - CQ_PHIBAR ** (-1.0 - CQ_ALPHA))

    def relax(self, u, rho, S, h, sweeps):
        """Red-black sweeps, each cell set to the root of its own equation (CQ: one Newton step)."""
        N = u.shape[0]
        i = torch.arange(N, device="cuda")
        colour = (i[:, None, None] + i[None, :, None] + i[None, None, :]) & 1
        for s in range(2 * sweeps):
            wn = _lap(self.w(u)) + 6.0 * self.w(u)
            if self.kind == "cq":
                x = CQ_PHIBAR + u / self.c2
                dr = -6.0 / (h * h) - self.pot * (1.0 + CQ_ALPHA) * x ** (-2.0 - CQ_ALPHA) / self.c2
                v = u - (self.N(u, rho, h) - S) / dr
            else:
                v = self._root(wn, rho, S, h, u)
            u = torch.where(colour == (s & 1), v, u)
        return u

    def _root(self, wn, rho, S, h, u):
        """The positive root of x^m + p x + q with q < 0 (largest where there are several), m = n + 2 (f(R)) or 3:
        Newton from above, where the polynomial is convex and rising."""
        if self.kind == "fr":
            al, m = h * h / (6.0 * self.c2), self.n + 2
            p, q = al * (self.om_a * (rho - 1.0) + self.K0 - S) - wn / 6.0, torch.full_like(wn, -al * self.K)
        else:
            g, m = self.c2 * self.xi ** 2 / (h * h), 3
            p, q = rho * self.r3 - 1.0 + 12.0 * g, -2.0 * g * wn + 2.0 * self.xi ** 2 * S
        sign = -torch.sign(q)
        q = -q.abs()
        # bound: x^m = -p x - q <= 2 max(|p| x, |q|)
        x = torch.maximum((2.0 * p.clamp(max=0.0).abs()) ** (1.0 / (m - 1)), (2.0 * q.abs()) ** (1.0 / m))
        for _ in range(60):
            x = x - (x ** m + p * x + q) / (m * x ** (m - 1) + p)
        return x * sign if self.kind == "sym" else x

    def solve(self, rho):
        """The solution of N(u) = 0 for a density of mean 1."""
        if self.kind == "fr":
            e = 1.0 / (self.n + 1)
            src = self.om_a * (rho - 1.0) + self.K0
            w = torch.minimum(torch.full_like(rho, self.ubar), self.K / src) ** (self.n + 1)
            for _ in range(60):
                F = -self.c2 * _lap(w) + src - self.K * w ** -e
                step = _pcg(self.c2, self.K * e * w ** (-e - 1.0), -F, 1e-4)
                big = float((step / w).abs().max())
                w = w * torch.exp((step / w).clamp(-2.0, 2.0)) if big > 1e-2 else w + step
                if big < 1e-11:
                    break
            return w ** e
        if self.kind == "sym":
            u = torch.ones_like(rho)
            for _ in range(60):
                F = -self.c2 * _lap(u) + self.ms * ((rho * self.r3 - 1.0) * u + u ** 3)
                step = _pcg(self.c2, self.ms * (rho * self.r3 - 1.0 + 3.0 * u * u), -F, 1e-4)
                u = u + step
                if float(step.abs().max()) < 1e-11 * self.ubar:
                    break
            return u
        u = torch.zeros_like(rho)
        N = u.shape[0]
        kx, ky, kz = (4.0 * torch.sin(0.5 * k) ** 2 for k in _k(N))
        K2 = kx + ky + kz + self.pot * (1.0 + CQ_ALPHA) * CQ_PHIBAR ** (-2.0 - CQ_ALPHA) / self.c2
        for _ in range(30):
            step = torch.fft.irfftn(torch.fft.rfftn(self.N(u, rho)) / K2, s=(N, N, N))
            u = u + step
            if float(step.abs().max()) < 1e-14 * float(u.abs().max()):
                break
        return u

    def potential(self, u):
        """The fifth-force potential about its background value: F = grad of it."""
        if self.kind == "fr":
            return -0.5 * self.c2 * (self.w(u) - self.ubar ** (self.n + 1))
        if self.kind == "sym":
            return -3.0 * self.xi ** 2 * OM * self.c2 / A_STAR ** 3 * (u * u - self.ubar ** 2)
        return -CQ_BETA * u


def _lap(u):
    s = -6.0 * u
    for d in range(3):
        s += torch.roll(u, 1, d)
        s += torch.roll(u, -1, d)
    return s


def _interp(x, d):
    """Linear interpolation of cell averages to half-size cells along axis d."""
    a, b = 0.75 * x + 0.25 * torch.roll(x, 1, d), 0.75 * x + 0.25 * torch.roll(x, -1, d)
    shape = list(x.shape)
    shape[d] *= 2
    return torch.stack([a, b], dim=d + 1).reshape(shape)


def _interp_t(x, d):
    """Half the transpose of _interp."""
    shape = list(x.shape)
    shape[d:d + 1] = [shape[d] // 2, 2]
    a, b = x.reshape(shape).unbind(d + 1)
    return 0.5 * (0.75 * (a + b) + 0.25 * (torch.roll(a, -1, d) + torch.roll(b, 1, d)))


def _vcycle(ops, l, b):
    k, m = ops[l]
    dinv = 0.85 / (6.0 * k + m)
    x = dinv * b
    sweeps = 1 if l + 1 < len(ops) else 12
    for _ in range(sweeps):
        x = x + dinv * (b + k * _lap(x) - m * x)
    if l + 1 < len(ops):
        r = b + k * _lap(x) - m * x
        for d in range(3):
            r = _interp_t(r, d)
        e = _vcycle(ops, l + 1, r)
        for d in range(3):
            e = _interp(e, d)
        x = x + e
        for _ in range(2):
            x = x + dinv * (b + k * _lap(x) - m * x)
    return x


def _pcg(kappa, m, b, rtol, most=200):
    """(-kappa Lap + m) x = b by conjugate gradients with a symmetric multigrid cycle as the preconditioner."""
    ops, n = [(kappa, m)], m.shape[0]
    while n % 2 == 0 and n > 4:
        n //= 2
        k, c = ops[-1]
        ops.append((k / 4.0, c.reshape(n, 2, n, 2, n, 2).mean((1, 3, 5))))
    x, r = torch.zeros_like(b), b
    end = rtol * float(torch.linalg.vector_norm(b))
    p = rz = None
    for _ in range(most):
        if float(torch.linalg.vector_norm(r)) <= end:
            break
        z = _vcycle(ops, 0, r)
        new = float((r * z).sum())
        p = z if p is None else z + (new / rz) * p
        rz = new
        Ap = m * p - kappa * _lap(p)
        t = rz / float((p * Ap).sum())
        x, r = x + t * p, r - t * Ap
    return x


def _cic(pos, N):
    """The 8 cells around each particle and their weights."""
    x = pos.double().remainder(float(N)) - 0.5
    c0 = torch.floor(x)
    f = x - c0
    c0 = c0.long()
    for a in range(2):
        for b in range(2):
            for d in range(2):
                o = (a, b, d)
                i, j, k = ((c0[:, t] + o[t]).remainder(N) for t in range(3))
                w = torch.ones_like(f[:, 0])
                for t in range(3):
                    w = w * (f[:, t] if o[t] else 1.0 - f[:, t])
                yield (i * N + j) * N + k, w


def _deposit(pos, N):
    rho = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
    for cell, w in _cic(pos, N):
        rho.index_add_(0, cell, w)
    return (rho * (N ** 3 / pos.shape[0])).reshape(N, N, N)


def _interpolate(mesh, pos):
    out = torch.zeros(pos.shape[0], dtype=torch.float64, device="cuda")
    for cell, w in _cic(pos, mesh.shape[0]):
        out += w * mesh.reshape(-1)[cell]
    return out


def _force(pot, pos):
    return torch.stack([_interpolate(0.5 * (torch.roll(pot, -1, d) - torch.roll(pot, 1, d)), pos) for d in range(3)], 1)


def _newton_potential(rho, coef):
    N = rho.shape[0]
    kx, ky, kz = (4.0 * torch.sin(0.5 * k) ** 2 for k in _k(N))
    K2 = kx + ky + kz
    K2[0, 0, 0] = 1.0
    f = torch.fft.rfftn(coef * (rho / rho.mean() - 1.0)) / -K2
    f[0, 0, 0] = 0.0
    return torch.fft.irfftn(f, s=(N, N, N))


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return [_Model(m).solve(_mean1(_density(m["N"], m["sigma"], seed + 7 * i))) for i, m in enumerate(_batch_members(c))]
    N, kind = c["N"], c["kind"]
    if kind == "deposit":
        return _deposit(_particles(N, c["M"], c["sigma"], seed)[0], N)
    if kind == "poisson":
        return _newton_potential(_density(N, c["sigma"], seed).double(), 1.5 * OM)
    if kind == "pm":
        return _exact_step(c, seed)
    m = _Model(c)
    if kind == "solve":
        u = m.solve(_mean1(_density(N, c["sigma"], seed)))
        if c["model"] != "cq":
            return {"field": u}
        return {"field": u - u.mean(), "force": _force(m.potential(u), _particles(N, c["M"], c["sigma"], seed + 1)[0])}
    if kind == "gather":
        return _force(m.potential(_field(c, seed + 1)), _particles(N, c["M"], c["sigma"], seed)[0])
    if kind == "twogrid":
        rho = _mean1(_density(N, c["sigma"], seed))
        mean8 = lambda x: x.reshape(N // 2, 2, N // 2, 2, N // 2, 2).mean((1, 3, 5))
        u = m.relax(_field(c, seed + 1), rho, 0.0, 1.0, 2)
        RuH, rhoH = mean8(u), mean8(rho)
        S = m.N(RuH, rhoH, 2.0) - mean8(m.N(u, rho))
        uH = m.relax(RuH, rhoH, S, 2.0, 2)
        e = uH - RuH
        for d in range(3):
            e = _interp(e, d)
        v = u + e
        if c["model"] == "fr":
            v = torch.where(v > 0.0, v, 0.5 * u)
        v = m.relax(v, rho, 0.0, 1.0, 2)
        return {"u": v, "uH": uH, "d": m.N(v, rho)}
    # gradient: J^T lambda = g, then through the density's normalisation and K ~ |fR0|^{1/(n+1)}
    rho = _density(N, c["sigma"], seed).double()
    mean = rho.mean()
    u = m.solve(rho / mean)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    g = torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64)
    if c["model"] == "fr":
        np1 = m.n + 1
        lam = _pcg(m.c2, m.K / (np1 * u ** (m.n + 2)), g / (np1 * u ** m.n), 1e-13)
        gd, gt = -m.om_a * lam, (lam * (m.K / (np1 * u))).sum()
    else:
        lam = _pcg(m.c2, m.ms * (rho / mean * m.r3 - 1.0 + 3.0 * u * u), -g, 1e-13)
        gd, gt = m.ms * m.r3 * u * lam, torch.zeros((), dtype=torch.float64)
    return {"field": u, "grad_rho": (gd - (gd * rho).sum() / rho.sum()) / mean, "grad_log_fr0": gt}


def _mean1(rho):
    rho = rho.double()
    return rho / rho.mean()


def _exact_step(c, seed):
    N, a, da = c["N"], 0.9, 0.01
    pos, psi = _particles(N, c["M"], c["sigma"], seed, margin=0.3)
    mom = (psi * (a * a * _E(a))).double()
    rho = _deposit(pos, N)
    pot = -_newton_potential(rho, 1.5 * OM / a)
    drag, out = 0.0, {}
    if c["model"] != "lcdm":
        m = _Model(c, a)
        u = m.solve(rho)
        pot += m.potential(u)
        if c["model"] == "sym":
            drag = 9.0 * OM * m.xi ** 2 * math.sqrt(1.0 - m.r3) / a ** 4 * da * _interpolate(u, pos)[:, None]
        out["field"] = u
    mom = (mom * (1.0 - 0.5 * drag) + da / (a * _E(a)) * _force(pot, pos)) / (1.0 + 0.5 * drag)
    ah = a + 0.5 * da
    pos = (pos.double() + da / (ah ** 3 * _E(ah)) * mom).remainder(float(N))
    return dict(out, pos=pos, mom=mom)
