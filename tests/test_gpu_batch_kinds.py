"""Batches of every model on uneven meshes, called twice with other parameters and fields.

Each solve agrees with its own single solve to 1e-6 (both converge the same
equations to tol; the bound of test_batch.py).  The second call changes models'
parameters, densities and field buffers, which replays or recaptures the batch's
graph; its answers are the second call's.
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
MODELS = [dict(model=0, n=1), dict(model=1, a_star=0.5, xi=3.3e-4), dict(model=0, n=2), dict(model=0, n=0),
          dict(model=2, alpha=0.1, beta=-0.05, lam=1.440377, phibar=0.779528), dict(model=0, n=1)]
SIDES = [64, 32, 96, 32, 64, 160]


@pytest.mark.parametrize("nu1,nu2,sweeps", [(2, 2, 16), (3, 0, 8), (0, 3, 8)])
def test_batch_of_every_model(mg, nu1, nu2, sweeps):  # noqa: F811
    for call, fr0 in enumerate((1e-6, 5e-6)):
        prms = [mg.Params(box=float(N), max_cycles=60, nu1=nu1, nu2=nu2, coarse_sweeps=sweeps,
                          **({"fR0_abs": fr0} if m["model"] == 0 else {}), **m) for N, m in zip(SIDES, MODELS)]
        rhos = [cuda32(inputs.lognormal_density(N, 1.0 + 0.1 * call, seed=90 + i + 10 * call)) for i, N in enumerate(SIDES)]
        fields = [torch.full((N,) * 3, float("nan"), dtype=torch.float64, device="cuda") for N in SIDES]
        st = mg.solve_batch(prms, [1.0] * len(SIDES), rhos, fields, 1e-9, allow_unconverged=True)
        for N, p, r, f, s in zip(SIDES, prms, rhos, fields, st):
            ref = torch.full((N,) * 3, float("nan"), dtype=torch.float64, device="cuda")
            one = mg.solve_scalar(p, 1.0, r, ref, 1e-9, allow_unconverged=True)
            assert s.converged == one.converged  # without pre-smoothing CQ's mean does not get there
            a, b = f.cpu().numpy(), ref.cpu().numpy()
            if p.model == 2:  # the mean is not fixed by the equation (test_gpu_parity.py)
                a, b = a - a.mean(), b - b.mean()
            assert relL2(a, b) <= 1e-6
