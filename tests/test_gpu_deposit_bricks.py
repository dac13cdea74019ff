"""The brick-by-brick deposit gives the mesh of the particle-by-particle one, bit for bit.

M^3 particles in the order of a lattice are deposited by bricks; the same particles in
chunks that end between lattice planes one by one (integer sums, in any order).
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import cuda32, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# mesh sides below, at and above the window's; M with whole and partial bricks
@pytest.mark.parametrize("N", [16, 30, 40, 64, 96, 120])
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
    got = mg.deposit_cic(p, N)
    host = p.cpu().pin_memory()
    ref = mg.deposit_cic_host(host, torch.empty_like(p), N, chunks=7)
    assert (M ** 3 + 6) // 7 % (M * M) != 0
    assert torch.equal(got, ref)
    assert float(got.double().mean()) == pytest.approx(1.0, rel=1e-6)
