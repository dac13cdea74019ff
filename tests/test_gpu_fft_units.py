"""The FFT Poisson solve of a density in any units.

A power of two in the density's unit takes nothing from any value or sum (down to the
subnormals and up to float's limit), so the potential is the same to the last bit; and
white noise about means from 1e-30 to 1e38, small and large coefficients among them, is
compared with the 64-bit solution to 2e-5 of its maximum, as in test_gpu_fft.py.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from test_gpu_fft import offset_copy  # noqa: E402
from test_gpu_pm import mg, pm  # noqa: E402,F401  (fixtures)


def noise(N):
    return (1.0 + 0.5 * np.random.default_rng(N).uniform(-1.0, 1.0, size=(N, N, N))).astype(np.float32)


@pytest.mark.parametrize("N", [8, 16, 32, 64, 128, 256, 512])
def test_power_of_two_units(mg, N):  # noqa: F811
    rho = torch.from_numpy(noise(N)).cuda()
    ref = mg.poisson_fft(rho, 0.7)
    for k in (-100, -30, -19, 19, 30, 110, 126):
        phi = mg.poisson_fft(torch.ldexp(rho, torch.tensor(float(k), device="cuda")), 0.7)
        assert torch.equal(phi, ref), k


@pytest.mark.parametrize("N", [16, 64, 256])
@pytest.mark.parametrize("mean,coef", [(1e-30, 0.7), (1e-7, 0.7), (1e7, 0.7), (1.7e32, 0.7), (1.7e35, 0.7), (1e38, 0.7),
                                       (1e9, 1e-30), (1e-9, 1e30), (1.7e35, 1e-20)])
def test_any_mean(mg, pm, N, mean, coef):  # noqa: F811
    rho = (noise(N).astype(np.float64) * mean).astype(np.float32)
    ref = pm.poisson_fft(rho.astype(np.float64) / mean, 1.0)
    r = torch.from_numpy(rho).cuda()
    phi = mg.poisson_fft(r, coef)
    got = phi.cpu().numpy().astype(np.float64) / coef
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()
    out = offset_copy(r)
    mg.poisson_fft(offset_copy(r), coef, out)
    assert torch.equal(out, phi)


def test_units_change_from_call_to_call(mg):  # noqa: F811
    rho = torch.from_numpy(noise(64)).cuda()
    ref = mg.poisson_fft(rho, 0.7)
    for k in (100, 0, -90, 0):
        assert torch.equal(mg.poisson_fft(torch.ldexp(rho, torch.tensor(float(k), device="cuda")), 0.7), ref)


def test_few_particles(mg, pm):  # noqa: F811
    """Nearly all cells empty, and no cell with mass among the first rows."""
    N = 64
    rho = np.zeros((N, N, N), np.float32)
    i = np.random.default_rng(5).integers(N // 2, N, size=(3, 40))
    rho[i[0], i[1], i[2]] = 1.7e35
    ref = pm.poisson_fft(rho.astype(np.float64) / 1.7e35, 0.7)
    phi = mg.poisson_fft(torch.from_numpy(rho).cuda(), 0.7).cpu().numpy()
    assert np.abs(phi - ref).max() <= 2e-5 * np.abs(ref).max()
