"""Deposit and gather by bricks of particles far from their bricks, and what surrounds them.

Arrays in lattice order of which a fraction is anywhere: the bricks that are asked keep
the particles that decide (checked here with the kernels' rule), so that these arrays go
by bricks, and their windows miss up to all of the other particles -- fewer than the list
of a CTA holds (256 in the deposit, 512 in the gather), more, and all.  The same
particles in chunks that end between lattice planes go one by one.  Tolerances as in
test_gpu_deposit_bricks.py (the same bits) and test_gpu_gather_bricks.py (1e-6).
"""
import numpy as np
import pytest

from paper_2110_00328_gb300 import inputs
from test_gpu_parity import cuda32, cuda64, mg  # noqa: F401  (mg: the fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def asked(M):
    """Pairs of particles (first and middle of 256 bricks of 8 x 8 x 32) and their distance in the lattice."""
    nbj, nbk = -(-M // 8), -(-M // 32)
    b = np.arange(256) * (nbj * nbj * nbk) // 256
    o = np.stack([b // nbk // nbj * 8, b // nbk % nbj * 8, b % nbk * 32], axis=1)
    d = np.minimum([4, 4, 8], M - 1 - o)
    flat = lambda x: (x[:, 0] * M + x[:, 1]) * M + x[:, 2]
    return flat(o), flat(o + d), d


def in_order(pos, N, M):
    """How many of the 256 say that the array is a lattice's."""
    a, b, d = asked(M)
    o = pos[b].astype(np.float64) - pos[a] - d * (N / M)
    return int((np.abs(o - N * np.rint(o / N)) < 12.0).all(axis=1).sum())


def displaced(N, M, fraction):
    rng = np.random.default_rng(M + N)
    pos = inputs.zeldovich_positions(N, seed=N, sigma=1.0, npart_side=M).astype(np.float32)
    far = rng.random(M ** 3) < fraction
    a, b, _ = asked(M)
    far[a] = far[b] = False
    pos[far] = rng.uniform(0.0, N, size=(int(far.sum()), 3))
    assert in_order(pos, N, M) >= 160
    return cuda32(pos)


@pytest.mark.parametrize("N,M", [(64, 192), (98, 200), (160, 193), (150, 192)])
@pytest.mark.parametrize("fraction", [0.0, 0.08, 0.6, 1.0])
def test_deposit(mg, N, M, fraction):  # noqa: F811
    p = displaced(N, M, fraction)
    got = mg.deposit_cic(p, N)
    assert (M ** 3 + 6) // 7 % (M * M) != 0
    assert torch.equal(got, mg.deposit_cic_host(p.cpu().pin_memory(), torch.empty_like(p), N, chunks=7))


# 16-byte rows and not; N M^3 >= 8.4e8, below which the gather goes by singles
@pytest.mark.parametrize("N,M", [(98, 224), (128, 200), (160, 193), (150, 192)])
@pytest.mark.parametrize("fraction", [0.0, 0.08, 0.6, 1.0])
def test_gather(mg, N, M, fraction):  # noqa: F811
    assert N * M ** 3 >= 8.4e8
    p = displaced(N, M, fraction)
    prm = mg.Params(box=float(N))
    field = cuda64(1.0 + 0.1 * np.random.default_rng(N).uniform(size=(N, N, N)))
    got = mg.gather_force(prm, 1.0, field, p)
    host = torch.empty((M ** 3, 3), dtype=torch.float32, pin_memory=True)
    mg.gather_force_host(prm, 1.0, field, p, torch.empty_like(p), host, chunks=7)
    torch.cuda.synchronize()
    ref = host.cuda()
    assert float((got - ref).abs().max()) <= 1e-6 * float(ref.abs().max())


@pytest.mark.parametrize("chunks", [1, 4])
def test_host_chunks_of_whole_planes(mg, chunks):  # noqa: F811
    """Chunks that are lattices themselves: each is asked for its own order."""
    N, M = 96, 256
    p = displaced(N, M, 0.05)
    assert torch.equal(mg.deposit_cic(p, N), mg.deposit_cic_host(p.cpu().pin_memory(), torch.empty_like(p), N, chunks=chunks))


@pytest.mark.parametrize("ordered", [True, False])
def test_calls_one_after_another(mg, ordered):  # noqa: F811
    """Calls on other particles and fields back to back: none sees what another one left, whichever kernel works."""
    N, M = 128, 192
    rng = np.random.default_rng(0)
    prm = mg.Params(box=float(N))
    sets = []
    for fraction in (0.0, 0.3):
        p = displaced(N, M, fraction)
        if not ordered:
            p = p[torch.from_numpy(rng.permutation(M ** 3)).cuda()].contiguous()
        field = cuda64(1.0 + 0.1 * rng.uniform(size=(N, N, N)))
        rho = mg.deposit_cic_host(p.cpu().pin_memory(), torch.empty_like(p), N, chunks=7)
        force = mg.gather_force(prm, 1.0, field, p)
        torch.cuda.synchronize()
        sets.append((p, field, rho, force))
    got = []
    for _ in range(4):
        for p, field, _, _ in sets:
            got.append((mg.deposit_cic(p, N), mg.gather_force(prm, 1.0, field, p)))
    for i, (r, f) in enumerate(got):
        assert torch.equal(r, sets[i % 2][2]) and torch.equal(f, sets[i % 2][3])


@pytest.mark.parametrize("ordered", [True, False])
def test_under_capture(mg, ordered):  # noqa: F811
    """A captured deposit, gather and Poisson solve, replayed on other particles in the same buffers."""
    N, M = 128, 192
    p = displaced(N, M, 0.0)
    other = displaced(N, M, 0.3)
    if not ordered:
        other = other[torch.from_numpy(np.random.default_rng(0).permutation(M ** 3)).cuda()].contiguous()
    field = cuda64(1.0 + 0.1 * np.random.default_rng(N).uniform(size=(N, N, N)))
    prm = mg.Params(box=float(N))
    rho, phi = (torch.empty((N, N, N), dtype=torch.float32, device="cuda") for _ in range(2))
    force = torch.empty_like(p)

    def calls():
        mg.deposit_cic(p, N, rho)
        mg.gather_force(prm, 1.0, field, p, 1.0, force)
        mg.poisson_fft(rho, 0.7, phi)

    calls()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    p.copy_(other)
    g.replay()
    torch.cuda.synchronize()
    got = [x.clone() for x in (rho, force, phi)]
    calls()
    for a, b in zip(got, (rho, force, phi)):
        assert torch.equal(a, b)
