"""The real-row FFT Poisson solve: every mode, the Nyquist ones included, and unaligned meshes.

White noise puts the same power in all modes.  The transforms' rounding is a few
2^-24 of the largest mode sum per pass (log2 N butterflies, six passes), so phi is
compared with the 64-bit solution to 2e-5 of its maximum, as in test_gpu_pm.py;
a single z-Nyquist plane wave, whose solution is -coef delta / 4, to 1e-6.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from test_gpu_pm import mg, pm  # noqa: E402,F401  (fixtures)

SIDES = [8, 16, 32, 64, 128]


def offset_copy(x):
    """The same mesh one float past an aligned address."""
    buf = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)
    v = buf[1:].view(x.shape)
    v.copy_(x)
    return v


@pytest.mark.parametrize("N", SIDES)
def test_white_noise_and_alignment(mg, pm, N):  # noqa: F811
    rho = (1.0 + 0.5 * np.random.default_rng(N).uniform(-1.0, 1.0, size=(N, N, N))).astype(np.float32)
    ref = pm.poisson_fft(rho.astype(np.float64), 0.7)
    r = torch.from_numpy(rho).cuda()
    phi = mg.poisson_fft(r, 0.7)
    assert np.abs(phi.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
    out = offset_copy(r)
    mg.poisson_fft(offset_copy(r), 0.7, out)
    assert torch.equal(out, phi)


@pytest.mark.parametrize("N", SIDES)
@pytest.mark.parametrize("axes", [(2,), (0, 2), (0, 1, 2)])
def test_nyquist_plane_wave(mg, N, axes):  # noqa: F811
    s = torch.ones((N, N, N), dtype=torch.float32, device="cuda")
    alt = 1.0 - 2.0 * (torch.arange(N, device="cuda") & 1).float()
    for d in axes:
        s = s * alt.view([-1 if i == d else 1 for i in range(3)])
    phi = mg.poisson_fft(1.0 + 0.5 * s, 1.5)
    assert float((phi + 1.5 * 0.5 * s / (4.0 * len(axes))).abs().max()) <= 1e-6
