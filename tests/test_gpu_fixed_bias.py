"""Rounding in the fixed-point passes goes both ways.

What always rounds one way adds up in a transform: at index 0 of the spectrum,
or at x = 0 or y = 0 of the field. Over 60 fields the mean error of every
coefficient and every point is compared with its standard error, taken from the
mean square of all errors: errors without a preferred sign give values of a few
(4.5 for the largest of 8192 normal ones; a real coefficient's own spread is at
most sqrt(2) of the mean's, a matvec's errors follow 1/h, at most twice here), so
10 leaves no room for chance. Rounded upwards, the spectra reach 30 to 150, with
sums rounded downwards the operator 12 to 80.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
COUNT, BOUND = 60, 10.0
LD = np.longdouble
TWO_PI = 2 * LD("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(LD).nmant < 60:
        pytest.skip("no extended precision here")


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def largest(errors):
    """The largest mean error in units of its standard error."""
    e = np.array(errors)
    return float(np.abs(e.mean(0)).max() / np.sqrt((np.abs(e) ** 2).mean() / len(e)))


@pytest.mark.parametrize("Nx,Ny", [(64, 8), (256, 8), (8, 256), (512, 16), (8, 1024)])
def test_transforms_have_no_preferred_sign(Nx, Ny):
    from paper_2306_09731_gb300.sgn import Solver
    rng = np.random.default_rng(Nx + Ny)
    s = Solver(Nx, Ny, 3.0, 5.0)
    forward, inverse = [], []
    for _ in range(COUNT):
        f = rng.standard_normal((Ny, Nx))
        F = np.fft.rfft2(f.astype(LD))
        forward.append((s.fft2(dev(f)).cpu().numpy() - F).astype(np.complex128))
        G = F.astype(np.complex128)
        inverse.append((s.ifft2(dev(G)).cpu().numpy()
                        - np.fft.irfft2(G.astype(np.clongdouble), s=f.shape)).astype(np.float64))
    s.close()
    assert largest(forward) <= BOUND
    assert largest(inverse) <= BOUND


@pytest.mark.parametrize("Nx,Ny", [(256, 16), (1024, 8), (16, 256), (8, 1024)])
@pytest.mark.parametrize("kind", ["noise", "smooth"])
def test_operator_has_no_preferred_sign(Nx, Ny, kind):
    from paper_2306_09731_gb300.sgn import Solver
    rng = np.random.default_rng(Nx + Ny)
    Lx, Ly = 0.1 * Nx, 0.1 * Ny
    y, x = np.mgrid[0:Ny, 0:Nx]
    X, Y = 2 * np.pi * x / Nx, 2 * np.pi * y / Ny
    kx = TWO_PI * np.arange(Nx // 2 + 1) / LD(Lx)
    m = np.fft.fftfreq(Ny, 1.0 / Ny)
    m[Ny // 2], kx[-1] = 0.0, 0.0
    waves = kx[None, :], (TWO_PI * m / LD(Ly))[:, None]
    s = Solver(Nx, Ny, Lx, Ly)
    errors = []
    for _ in range(COUNT):
        p = rng.uniform(0.0, 2 * np.pi, 5)
        h = 1.0 + 0.3 * np.cos(X + p[0]) * np.cos(Y + p[1])
        if kind == "noise":
            sg = rng.standard_normal(h.shape)
        else:
            sg = 1.0 + np.cos(X + p[2]) + 0.5 * np.sin(2 * X + Y + p[3]) + 0.2 * np.cos(3 * X - 2 * Y + p[4])
        H, S = h.astype(LD), np.fft.rfft2(sg.astype(LD))
        ref = 3 * sg.astype(LD) / H ** 3
        for k in waves:
            g = np.fft.irfft2(1j * k * S, s=h.shape) / H
            ref = ref - np.fft.irfft2(1j * k * np.fft.rfft2(g), s=h.shape)
        errors.append((s.elliptic_apply(dev(h), dev(sg)).cpu().numpy() - ref).astype(np.float64))
    s.close()
    assert largest(errors) <= BOUND
