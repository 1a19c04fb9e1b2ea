"""Derivatives of small variations on a large mean, FP64 transforms in fixed point.

The field holds whole numbers below 2^18 plus a mean of up to 2^34, which FP64
stores and sums exactly: the mean adds nothing to the derivative, and no
rounding either. Error against extended precision: the spectrum's noise
(test_gpu_fixed.py's bound for a 2D transform, of the variations' norm) times
the largest wavenumber, and the same bound once more, of the derivative, for
the way back.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOUND = 5.6e-16


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("Nx,Ny", [(8, 8), (256, 64), (64, 1024), (4096, 16), (16, 4096)])
@pytest.mark.parametrize("mean", [0.0, 2.0 ** 20, -2.0 ** 34])
def test_a_mean_costs_the_derivative_nothing(Nx, Ny, mean):
    from paper_2306_09731_gb300.sgn import Solver
    y, x = np.mgrid[0:Ny, 0:Nx]
    q = np.round(2.0 ** 17 * (np.cos(2 * np.pi * x / Nx) + 0.5 * np.sin(2 * np.pi * (2 * y / Ny + x / Nx))
                              + 0.25 * np.cos(2 * np.pi * 3 * y / Ny)))
    s = Solver(Nx, Ny, 3.0, 5.0)
    fx, fy = (t.cpu().numpy() for t in s.derivative(torch.tensor(q + mean, device="cuda")))
    s.close()
    F = np.fft.rfft2(q.astype(np.longdouble))
    two_pi = 2 * np.longdouble("3.14159265358979323846264338327950288")
    kx = two_pi / 3 * np.arange(Nx // 2 + 1)
    kx[-1] = 0.0
    m = np.fft.fftfreq(Ny, 1.0 / Ny)
    m[Ny // 2] = 0.0
    ky = two_pi / 5 * m
    for got, k in ((fx, kx[None, :]), (fy, ky[:, None])):
        ref = np.fft.irfft2(1j * k * F, s=q.shape)
        tol = BOUND * (np.linalg.norm(q) * float(np.abs(k).max()) + float(np.sqrt((ref ** 2).sum())))
        assert float(np.sqrt(((got - ref) ** 2).sum())) <= tol


def test_an_infinite_mean_is_seen():
    from paper_2306_09731_gb300.sgn import Solver
    s = Solver(64, 32, 3.0, 5.0)
    for bad in (float("inf"), float("nan")):
        f = torch.full((32, 64), bad, dtype=torch.float64, device="cuda")
        for d in s.derivative(f):
            assert bool(torch.isnan(d).all())
    s.close()
