"""The FP64 transforms on 64-bit fixed point (csrc/fixed.cuh, csrc/sgn_fx.cuh).

Reference: numpy transforms in extended precision where the platform has it
(longdouble), so that the reference's rounding does not count. Bound of the
relative 2-norm error of one 2D transform: each of the two passes rounds its
result to FP64 (2^-53 at most, 2^-53/sqrt 3 rms) and adds the fixed-point noise
of one transform, at most 1.7e-16 for every length up to 4096: 2 (1.7e-16 +
1.1e-16) = 5.6e-16 at worst.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

BOUND = 5.6e-16
SIZES = [(8, 8), (16, 8), (8, 64), (32, 512), (128, 16), (256, 1024), (2048, 8), (8, 4096), (4096, 16)]


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def rel(a, r):
    d = np.abs(a.astype(np.clongdouble) - r.astype(np.clongdouble))
    return float(np.sqrt((d ** 2).sum() / (np.abs(r) ** 2).sum()))


def field(kind, Nx, Ny):
    rng = np.random.default_rng(Nx * 7 + Ny)
    y, x = np.mgrid[0:Ny, 0:Nx]
    if kind == "noise":
        return rng.standard_normal((Ny, Nx))
    if kind == "integers":  # few significant bits: every low limb pattern occurs
        return rng.integers(-8, 9, (Ny, Nx)).astype(np.float64)
    if kind == "spike":
        f = np.zeros((Ny, Nx))
        f[Ny // 3, Nx // 5] = -3.0
        return f
    if kind == "range":  # rows of very different size, huge and tiny
        return rng.standard_normal((Ny, Nx)) * 10.0 ** (2.0 * (y // 2) / Ny)
    return 1.0 + 1e-6 * np.sin(2 * np.pi * (x / Nx + 2 * y / Ny))  # small on large


@pytest.mark.parametrize("Nx,Ny", SIZES)
@pytest.mark.parametrize("kind", ["noise", "integers", "spike", "range", "offset"])
@pytest.mark.parametrize("scale", [1.0, 1e250, 1e-250])
def test_transforms_against_extended_precision(Nx, Ny, kind, scale):
    from paper_2306_09731_gb300.sgn import Solver
    f = field(kind, Nx, Ny) * scale
    s = Solver(Nx, Ny, 3.0, 5.0)
    F = s.fft2(dev(f)).cpu().numpy()
    ref = np.fft.rfft2(f.astype(np.longdouble) / scale)
    assert rel(F / scale, ref) <= BOUND
    G = ref.astype(np.complex128)
    back = s.ifft2(dev(G * scale)).cpu().numpy()
    want = np.fft.irfft2((G * scale).astype(np.clongdouble) / scale, s=f.shape)
    assert rel(back / scale, want) <= BOUND
    s.close()


@pytest.mark.parametrize("Nx,Ny", [(64, 32), (2048, 16), (16, 2048)])
def test_small_variations_keep_their_accuracy(Nx, Ny):
    """The derivative of 1 + 1e-6 sin: its rounding error is that of the input
    (2^-53 of 1 per point, times the largest wavenumber) and not larger."""
    from paper_2306_09731_gb300.sgn import Solver
    f = field("offset", Nx, Ny)
    s = Solver(Nx, Ny, 3.0, 5.0)
    fx, fy = (t.cpu().numpy() for t in s.derivative(dev(f)))
    s.close()
    F = np.fft.rfft2(f.astype(np.longdouble))
    kx = 2 * np.pi * np.arange(Nx // 2 + 1) / 3.0
    kx[-1] = 0.0
    m = np.fft.fftfreq(Ny, 1.0 / Ny)
    m[Ny // 2] = 0.0
    ky = 2 * np.pi * m / 5.0
    for got, k in ((fx, kx[None, :]), (fy, ky[:, None])):
        ref = np.fft.irfft2(1j * k * F, s=f.shape)
        # noise of the spectrum, in the physical norm: BOUND * |f - 1| and the
        # rounding of the mean's own row and column sums (2^-53), times max |k|
        tol = (BOUND * np.linalg.norm(f - 1.0) + 2.0 ** -53 * np.sqrt(f.size)) * np.abs(k).max()
        assert float(np.sqrt(((got - ref) ** 2).sum())) <= tol


def test_zero_and_nonfinite_inputs():
    from paper_2306_09731_gb300.sgn import Solver
    s = Solver(64, 32, 3.0, 5.0)
    z = torch.zeros((32, 64), dtype=torch.float64, device="cuda")
    assert int(torch.count_nonzero(torch.view_as_real(s.fft2(z)))) == 0
    for bad in (float("nan"), float("inf"), -float("inf")):
        f = z.clone()
        f[5, 7] = bad
        assert bool(torch.isnan(torch.view_as_real(s.fft2(f))).all())
        h = torch.ones_like(z)
        F = s.fft2(h)
        F[3, 4] = bad
        assert bool(torch.isnan(s.ifft2(F)).all())
    s.close()
