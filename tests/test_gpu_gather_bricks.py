"""The brick-by-brick gather gives the particle-by-particle one's forces.

M^3 particles in the order of a lattice are gathered by bricks; the same particles in
chunks that end between lattice planes one by one.  Both form the same sums of the same
cells in the same order, up to where the compiler fuses a product into a sum: bounded by
a few roundings of the largest difference, 1e-6 of the largest force component.
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import cuda32, cuda64, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# mesh sides below, at and above the window's, multiples of four (16-byte rows) and not;
# M with whole and partial bricks
@pytest.mark.parametrize("N", [30, 48, 50, 64, 98, 120])
@pytest.mark.parametrize("M", [185, 192])
@pytest.mark.parametrize("kind", ["lattice", "random", "clump", "two clumps", "wrap"])
def test_bricks_equal_singles(mg, N, M, kind):  # noqa: F811
    rng = np.random.default_rng(M + N)
    if kind == "lattice":
        pos = inputs.zeldovich_positions(N, seed=N, sigma=1.5, npart_side=M)
    elif kind == "random":
        pos = rng.uniform(0.0, N, size=(M ** 3, 3))
    elif kind == "clump":  # every particle in one cell, at its corners, faces and centre
        pos = 3.0 + 0.5 * rng.integers(0, 3, size=(M ** 3, 3))
    elif kind == "two clumps":  # a mean between them, far from both
        pos = 0.1 * N + 0.5 * N * rng.integers(0, 2, size=(M ** 3, 1)) + rng.uniform(-1.0, 1.0, size=(M ** 3, 3))
    else:
        pos = inputs.zeldovich_positions(N, seed=N, sigma=1.5, npart_side=M).astype(np.float64) + N * rng.integers(-2, 3, size=(M ** 3, 3))
    p = cuda32(pos)
    prm = mg.Params(box=float(N))
    field = cuda64(1.0 + 0.1 * rng.uniform(size=(N, N, N)))
    got = mg.gather_force(prm, 1.0, field, p)
    host = torch.empty((M ** 3, 3), dtype=torch.float32, pin_memory=True)
    mg.gather_force_host(prm, 1.0, field, p, torch.empty_like(p), host, chunks=7)
    torch.cuda.synchronize()
    assert (M ** 3 + 6) // 7 % (M * M) != 0
    ref = host.cuda()
    assert float((got - ref).abs().max()) <= 1e-6 * float(ref.abs().max())
