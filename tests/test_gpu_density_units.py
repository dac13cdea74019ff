"""Every solve takes a density of any positive mean.

The density is rescaled to mean 1 by its sum, which stays in range up to float's own
limit.  A power of two in its unit changes no bit of the FP64 path; in the mixed path the
factor 1/mean of the residual's source nears float's smallest normal number at 2^124 (its
low part is then good to 2^-24 of it), which bounds the field by 1e-6.
"""
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def solve(mg, orc, key, N, k, precision):
    extra = dict(xi=3.3e-4) if key == "sym" else {}
    po, pg = both_params(orc, mg, key, box=float(N), precision=precision, **extra)
    rho = cuda32(inputs.lognormal_density(N, 0.8, seed=40 + N)).clamp(max=6.0)
    f = torch.full((N, N, N), float("nan"), dtype=torch.float64, device="cuda")
    st = mg.solve_scalar(pg, 1.0, torch.ldexp(rho, torch.tensor(float(k), device="cuda")), f, 1e-9)
    assert st.converged
    return f


@pytest.mark.parametrize("N", [32, 64])
@pytest.mark.parametrize("key", ["fr1", "sym"])
@pytest.mark.parametrize("k", [124, 100, -60])
def test_units_of_the_density(orc, mg, key, N, k):  # noqa: F811
    assert torch.equal(solve(mg, orc, key, N, k, mg.FP64), solve(mg, orc, key, N, 0, mg.FP64))
    a, b = (solve(mg, orc, key, N, x, mg.MIXED).cpu().numpy() for x in (k, 0))
    assert relL2(a, b) <= 1e-6
