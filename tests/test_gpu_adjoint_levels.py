"""The adjoint solve's level paths: split and natural finest levels, one- and two-cell
residual tiles, the one-block tail, and schedules without pre- or post-smoothing.

lambda is read back from dl/d delta and put into -c^2 Lap lambda + m lambda = sigma g
in FP64: the relative residual is what the call converged to (tol), plus the
rounding of the float-float residual that decided it (2^-44 of the largest term,
kappa (L - 6 lambda) and m lambda against sigma g: at most a few hundred here).
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-9


def lap(x):
    return sum(torch.roll(x, s, d) for d in range(3) for s in (1, -1)) - 6.0 * x


def solve(mg, pg, b, key, N, g):  # noqa: F811
    rho = cuda32(inputs.lognormal_density(N, 0.8, seed=70 + N))
    u = b["ubar"] / (1.0 + 0.3 * rho.double())
    grad, glog, st = mg.solve_adjoint(pg, 1.0, u.contiguous(), rho, g, tol=TOL)
    r = rho.double() / rho.double().mean()
    if key == "sym":
        m, sig, gam = b["msym"] * (r * 0.125 - 1.0 + 3.0 * u * u), -torch.ones_like(u), b["msym"] * 0.125 * u
        tq = torch.zeros_like(u)
    else:
        n = pg.n
        m, sig = b["K"] / ((n + 1) * u ** (n + 2)), 1.0 / ((n + 1) * u ** n)
        gam, tq = torch.full_like(u, -pg.omega_m), b["K"] / ((n + 1) * u)
    lam = grad / gam
    res = sig * g - (-b["c2"] * lap(lam) + m * lam)
    return float(res.norm() / (sig * g).norm()), glog, float((lam * tq).sum()), float((lam * tq).norm()), st


@pytest.mark.parametrize("N,extra", [(4, {}), (6, {}), (12, {}), (16, {}), (24, {}), (32, {}), (40, {}), (64, {}),
                                     (96, {}), (160, {}), (64, dict(nu1=0, nu2=2)), (64, dict(nu1=2, nu2=0)),
                                     (48, dict(levels=2)), (64, dict(levels=1, coarse_sweeps=300))])
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym"])
def test_solves_the_adjoint_equation(orc, mg, key, N, extra):  # noqa: F811
    po, pg = both_params(orc, mg, key, box=float(N), **(dict(xi=3.3e-4) if key == "sym" else {}), max_cycles=300, **extra)
    b = orc.background(po, N)
    g = torch.from_numpy(np.random.default_rng(N).normal(size=(N, N, N))).cuda()
    res, glog, want, scale, st = solve(mg, pg, b, key, N, g)
    assert st.converged and res <= 2.0 * TOL
    assert abs(glog - want) <= 1e-12 * scale * N ** 1.5  # rounding of N^3 terms of mixed sign


def test_scale_of_the_loss(orc, mg):  # noqa: F811
    po, pg = both_params(orc, mg, "fr1", box=64.0)
    b = orc.background(po, 64)
    g = torch.from_numpy(np.random.default_rng(3).normal(size=(64, 64, 64))).cuda()
    _, one, _, scale, _ = solve(mg, pg, b, "fr1", 64, g)
    _, small, _, _, _ = solve(mg, pg, b, "fr1", 64, g * 2.0 ** -40)
    assert abs(small * 2.0 ** 40 - one) <= 1e-9 * scale
