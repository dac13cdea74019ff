"""Coupled quintessence, mixed precision: the potential by its series and by the library,
on split, natural and untiled finest levels.

c~^2 runs from 9e6 (1 Mpc/h cells: the series, field ~1e-6 of c~^2 phibar) to 1
(cells of a Hubble length: powers throughout, field up to tenths of phibar).  In
between, the residual of the field's mean decays slowly (its mass is small against
the coarsest mesh's Laplacian, and no smoother reaches it), in the oracle as here;
so the oracle runs as many cycles, and the mixed solve's residual, recomputed by
the oracle, is at most twice its (or tol), and the field about its mean agrees with
the oracle's converged one to 1e-6 (the targets of test_gpu_parity.py, whose
docstring says why the mean is taken out).
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 1e-10


@pytest.mark.parametrize("N", [32, 40, 48, 64])
@pytest.mark.parametrize("cell", [1.0, 9.0, 12.0, 100.0, 2997.92458])  # Mpc/h: 9 and 12 straddle the series' limit
def test_cq_solve(orc, mg, N, cell):  # noqa: F811
    po, pg = both_params(orc, mg, "cq", box=N * cell, alpha=0.1, beta=-0.05, lam=1.440377, phibar=0.779528,
                         max_cycles=20)
    rho32 = inputs.lognormal_density(N, 1.2, seed=N).astype(np.float32)
    field = torch.full((N, N, N), float("nan"), dtype=torch.float64, device="cuda")
    st = mg.solve_scalar(pg, 1.0, cuda32(rho32), field, TOL, allow_unconverged=True)
    got = field.cpu().numpy()
    rho = rho32.astype(np.float64)
    rho = rho / rho.mean()
    d = orc.residual(po, got, rho)
    rms = lambda x: float(np.sqrt((x ** 2).mean()))
    eps = orc.solve(po, rho, tol=0.0, max_cycles=st.cycles, kind=orc.KIND_NEWTON).eps
    assert rms(d) <= 2.0 * max(TOL, eps) * orc.source_rms(po, rho) + 1e-14 * np.abs(got).max()
    ref = orc.solve(po, rho, tol=1e-12, max_cycles=80, kind=orc.KIND_NEWTON).u
    assert relL2(got - got.mean(), ref - ref.mean()) <= 1e-6
