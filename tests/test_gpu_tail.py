"""The one-block tail against one kernel per step: the same V-cycle.

One inner cycle with the tail and with it off (tail_cells < 0) from the background:
both apply the same single-precision arithmetic per cell in the same colour order,
so they differ by the rounding of differently associated sums, bounded as in
test_gpu_parity.py by 2e-5 of the deviation from the background after one cycle.
The sides put 4, 6, 8, 10, 12, 14 and 16 cells at the tail's first level, one and
two pairs a thread, whole and partial warps.
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [8, 12, 20, 24, 28, 32, 40, 56, 64])
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym", "cq"])
@pytest.mark.parametrize("nu1,nu2,sweeps", [(2, 2, 16), (1, 0, 3), (0, 1, 5)])
def test_tail_is_the_same_cycle(orc, mg, key, N, nu1, nu2, sweeps):  # noqa: F811
    extra = dict(xi=3.3e-4) if key == "sym" else {}
    rho = cuda32(inputs.lognormal_density(N, 1.0, seed=80 + N))
    out = []
    for tail in (0, -1):
        po, pg = both_params(orc, mg, key, box=float(N), nu1=nu1, nu2=nu2, coarse_sweeps=sweeps, max_cycles=1,
                             inner_cycles=1, tail_cells=tail, **extra)
        f = torch.full((N, N, N), float("nan"), dtype=torch.float64, device="cuda")
        st = mg.solve_scalar(pg, 1.0, rho, f, 1e-12, allow_unconverged=True)
        out.append((f.cpu().numpy() - (0.0 if key == "cq" else orc.background(po, N)["ubar"]), st.guarded))
    assert relL2(out[0][0], out[1][0]) <= 2e-5
    assert out[0][1] == out[1][1]
