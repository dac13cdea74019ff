"""The FP64 kernels' FP32-started roots and reciprocals against the oracle, cell by cell.

A sweep sets x to the root of x^m + p x + q.  With P the sum of the magnitudes of
p's terms, an FP64 evaluation of the polynomial is off by a few eps (x^m + P |x| +
|q|), and the root by that over |m x^{m-1} + p|.  The bound takes 32 eps: the
terms of p (nine roundings on either side), the neighbours' own errors, and the
red cells' black neighbours, which already carry theirs.
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda64, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EPS = np.finfo(np.float64).eps


def neighbours(w):
    return sum(np.roll(w, s, d) for d in range(3) for s in (1, -1))


def fields(n, decades, seed):
    """Density and field spread over 'decades' decades each (deep screening and voids)."""
    g = inputs.gaussian_field(n, seed=seed, sigma=1.0, cutoff=False)
    rho = np.exp(decades * g)
    return rho / rho.mean(), np.exp(-decades * inputs.gaussian_field(n, seed=seed + 1, sigma=1.0, cutoff=False))


# sides: below, at and past the 16-cell blocks, a remainder in both directions
@pytest.mark.parametrize("n", [4, 10, 16, 34])
@pytest.mark.parametrize("decades", [0.5, 3.0])
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym"])
@pytest.mark.parametrize("h", [1.0, 4.0])
def test_sweep_is_at_rounding(orc, mg, key, n, decades, h):  # noqa: F811
    po, pg = both_params(orc, mg, key, box=float(n * h))
    b = orc.background(po, int(n * h))
    rho, u0 = fields(n, decades, seed=50 + n)
    u0 = u0 * b["ubar"]
    if key == "sym":
        u0 = u0 * np.where(inputs.gaussian_field(n, seed=9) > 0.5, -1.0, 1.0)  # both branches
        S = 1e-2 * b["msym"] * inputs.gaussian_field(n, seed=52)
    else:
        S = 0.3 * b["K0"] * inputs.gaussian_field(n, seed=52)
    ref = orc.smooth(po, u0, rho, S=S, sweeps=1, h=h)
    u = cuda64(u0)
    mg.smooth(pg, 1.0, u, cuda64(rho), S=cuda64(S), sweeps=1, h=h)
    x = np.abs(ref)
    if key == "sym":
        g, m, k = b["c2"] * po.xi ** 2 / h ** 2, 3, 1
        L = 2.0 * g * neighbours(np.abs(ref) + np.abs(u0))
        p, P = rho * po.a_star ** 3 - 1.0 + 12.0 * g, rho * po.a_star ** 3 + 1.0 + 12.0 * g
        q = L + 2.0 * po.xi ** 2 * np.abs(S)
        num = x ** m + P * x + q
    else:
        al, k = h * h / (6.0 * b["c2"]), po.n + 1
        m = k + 1
        i = np.add.outer(np.add.outer(np.arange(n), np.arange(n)), np.arange(n)) & 1
        w = np.where(i == 0, ref, u0) ** k  # what the red cells saw
        L = np.where(i == 1, neighbours(w), neighbours(u0 ** k))
        p = al * (po.omega_m * (rho - 1.0) + b["K0"] - S) - L / 6.0
        P = al * (po.omega_m * (rho + 1.0) + b["K0"] + np.abs(S)) + L / 6.0
        num = x ** m + P * x + al * b["K"]
    bound = 32.0 * EPS * num / np.maximum(np.abs(m * x ** (m - 1) + p), 1e-300)
    err = np.abs(u.cpu().numpy() - ref)
    # the red cells also inherit the black ones' errors through their neighbour sum
    carried = neighbours(k * x ** (k - 1) * bound) * (2.0 * g if key == "sym" else x / 6.0)
    bound = bound + carried / np.maximum(np.abs(m * x ** (m - 1) + p), 1e-300)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("box_over_hubble", [0.05, 1.0])  # the series and the library power
@pytest.mark.parametrize("n", [10, 16])
def test_cq_step_and_residual(orc, mg, box_over_hubble, n):  # noqa: F811
    """One Newton step and the residual: the difference of the powers is a few eps of phibar^{-1-alpha}."""
    po, pg = both_params(orc, mg, "cq", box=n * 2997.92458 * box_over_hubble)
    b = orc.background(po, n)
    rho, _ = fields(n, 1.0, seed=60)
    u0 = 0.03 * inputs.gaussian_field(n, seed=61)
    pot = b["cq_pot"] * 0.5 ** -1.1
    ref = orc.smooth(po, u0, rho, sweeps=1, kind=orc.KIND_NEWTON)
    got = mg.smooth(pg, 1.0, cuda64(u0), cuda64(rho), sweeps=1).cpu().numpy()
    scale = np.abs(u0).max() * 12.0 + abs(b["cq_src"]) * rho.max() + pot
    assert np.abs(got - ref).max() <= 32.0 * EPS * scale
    d, _ = mg.residual(pg, 1.0, cuda64(u0), cuda64(rho))
    assert np.abs(d.cpu().numpy() - orc.residual(po, u0, rho)).max() <= 32.0 * EPS * scale


@pytest.mark.parametrize("n", [4, 12, 34])
def test_prolongation_shares_its_sums(orc, mg, n):  # noqa: F811
    """Every child against the oracle's; eight terms of at most |uH| + |RuH| each, plus the value corrected."""
    rng = np.random.default_rng(n)
    po, pg = both_params(orc, mg, "sym", box=float(2 * n))
    uh, uH, RuH = rng.normal(size=(2 * n,) * 3), rng.normal(size=(n,) * 3), rng.normal(size=(n,) * 3)
    ref, _ = orc.prolong_correct(po, uH, RuH, uh)
    got = mg.prolong_correct(pg, cuda64(uH), cuda64(RuH), cuda64(uh)).cpu().numpy()
    assert np.abs(got - ref).max() <= 16.0 * EPS * (np.abs(uH).max() + np.abs(RuH).max() + np.abs(uh).max())
