"""The adjoint's sums over the mesh carry FP64 rounding.

lambda is read back from dl/d delta, and the sums for dl/d ln|fR0| and for the density's
normalisation are formed again from it, exactly summed on the host.  A term differs by a
few roundings, at most 4 x 2^-53 of it and independent from cell to cell; the library's
sums are trees over a thread's cells, which add one 2^-53 of a partial sum a level, at
most 24 levels: together an error of standard deviation below 4 x 2^-53 |terms|_2.  The
bound is four times that.  The density's own sum, which the normalisation divides by, is
of two floats a thread, good to 2^-46.
"""
import math

import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import both_params, cuda32, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EPS = 2.0 ** -53


@pytest.mark.parametrize("N", [16, 64, 128])
@pytest.mark.parametrize("key", ["fr0", "fr1", "fr2", "sym"])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -60])
def test_sums_are_fp64(orc, mg, key, N, scale):  # noqa: F811
    po, pg = both_params(orc, mg, key, box=float(N), **(dict(xi=3.3e-4) if key == "sym" else {}), max_cycles=300)
    b = orc.background(po, N)
    rho = cuda32(inputs.lognormal_density(N, 0.8, seed=70 + N))
    u = (b["ubar"] / (1.0 + 0.3 * rho.double())).contiguous()
    g = scale * torch.from_numpy(np.random.default_rng(N).normal(size=(N, N, N))).cuda()
    grad, glog, _ = mg.solve_adjoint(pg, 1.0, u, rho, g, tol=1e-8)
    raw, _, _ = mg.solve_adjoint(pg, 1.0, u, rho, g, tol=1e-8, raw=True)
    if key != "sym":
        t = (grad / -pg.omega_m) * (b["K"] / ((pg.n + 1) * u))
        want = math.fsum(t.flatten().tolist())
        assert abs(glog - want) <= 16 * EPS * float(t.norm()) + 4 * EPS * abs(want)
    # grad_raw = (grad - shift) / mean, shift = sum(grad rho) / sum(rho); the mean of grad - mean grad_raw
    # averages the roundings of its cells
    r = rho.double()
    total = math.fsum(r.flatten().tolist())
    shift = math.fsum((grad - raw * (total / N ** 3)).flatten().tolist()) / N ** 3
    t = grad * r
    want = math.fsum(t.flatten().tolist()) / total
    assert abs(shift - want) <= 16 * EPS * (float(t.norm()) / total + float(grad.norm()) / N ** 3) + 2.0 ** -46 * abs(want)
