"""The one-block tail against one kernel per step: the same V-cycle.

tail_cells up to 4096 keeps the levels from a cluster of blocks (which starts at 20^3, or
on a finest level of at most tail_cells cells), so that k_tail32 runs from the first level
below the finest with at most tail_cells cells: 4, 6, 8, 10, 12, 14 and 16 a side here,
one and two pairs a thread, whole and partial warps.  Bounds as in test_gpu_tail.py: the
two differ by the rounding of differently associated sums, 2e-5 of the deviation from the
background after one cycle.
"""
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg, relL2  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# mesh, tail_cells, first tail level
FIRST = [(8, 64, 4), (12, 216, 6), (16, 512, 8), (20, 4096, 10), (24, 4096, 12), (28, 4096, 14), (32, 4096, 16),
         (40, 4096, 10), (48, 4096, 12), (56, 4096, 14), (64, 4096, 16)]


@pytest.mark.parametrize("N,cells,first", FIRST)
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym", "cq"])
@pytest.mark.parametrize("kw", [dict(), dict(nu1=1, nu2=0, coarse_sweeps=3), dict(nu1=0, nu2=1, coarse_sweeps=5)])
def test_one_block_tail_is_the_same_cycle(orc, mg, key, N, cells, first, kw):  # noqa: F811
    n = N // 2
    while n ** 3 > cells:
        n //= 2
    assert n == first and N ** 3 > cells
    extra = dict(xi=3.3e-4) if key == "sym" else {}
    rho = cuda32(inputs.lognormal_density(N, 1.0, seed=80 + N))
    out, launches = [], []
    for tail in (cells, -1):
        po, pg = both_params(orc, mg, key, box=float(N), max_cycles=1, inner_cycles=1, tail_cells=tail, **extra, **kw)
        f = torch.full((N, N, N), float("nan"), dtype=torch.float64, device="cuda")
        before = mg.launch_count()
        st = mg.solve_scalar(pg, 1.0, rho, f, 1e-12, allow_unconverged=True)
        launches.append(mg.launch_count() - before)
        out.append((f.cpu().numpy() - (0.0 if key == "cq" else orc.background(po, N)["ubar"]), st.guarded))
    assert launches[0] < launches[1]  # the tail's levels are one kernel
    assert relL2(out[0][0], out[1][0]) <= 2e-5
    assert out[0][1] == out[1][1]
