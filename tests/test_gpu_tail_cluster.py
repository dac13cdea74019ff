"""The clustered tail against one kernel per step: the same V-cycles.

Three inner cycles of one outer step with the tail and with it off (tail_cells < 0)
from the background: both apply the same single-precision arithmetic per cell in the
same colour order, so they differ by the rounding of differently associated sums,
bounded as in test_gpu_parity.py by 2e-5 of the deviation from the background.  The
sides put 8 to 32 cells on the cluster's first level, as the finest (natural and
split) and below it; the level counts leave two, three and all levels, so that the
second is the coarsest or not.
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def cycles(orc, mg, key, N, tail, **kw):
    extra = dict(xi=3.3e-4) if key == "sym" else {}
    rho = cuda32(inputs.lognormal_density(N, 1.0, seed=90 + N))
    po, pg = both_params(orc, mg, key, box=float(N), max_cycles=3, inner_cycles=3, tail_cells=tail, **extra, **kw)
    f = torch.full((N, N, N), float("nan"), dtype=torch.float64, device="cuda")
    st = mg.solve_scalar(pg, 1.0, rho, f, 1e-12, allow_unconverged=True)
    return f.cpu().numpy() - (0.0 if key == "cq" else orc.background(po, N)["ubar"]), st.guarded


@pytest.mark.parametrize("N", [8, 12, 16, 20, 24, 28, 32, 40, 48, 64])
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym", "cq"])
@pytest.mark.parametrize("kw", [dict(), dict(levels=2, coarse_sweeps=5), dict(levels=3, nu1=1, nu2=0), dict(nu1=0, nu2=1)])
def test_cluster_is_the_same_cycles(orc, mg, key, N, kw):  # noqa: F811
    if (N >> (kw.get("levels", 1) - 1)) % 2:
        pytest.skip("an odd coarsest side: no tail, and cells of one colour are neighbours across the boundary")
    a, b = (cycles(orc, mg, key, N, tail, **kw) for tail in (0, -1))
    assert relL2(a[0], b[0]) <= 2e-5
    assert a[1] == b[1]


@pytest.mark.parametrize("N", [16, 32, 64])
@pytest.mark.parametrize("key", ["fr1", "sym"])
def test_cluster_after_a_full_multigrid_start(orc, mg, key, N):  # noqa: F811
    a, b = (cycles(orc, mg, key, N, tail, fmg=1) for tail in (0, -1))
    assert relL2(a[0], b[0]) <= 2e-5
    assert a[1] == b[1]
