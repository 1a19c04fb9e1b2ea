"""Sizes around the lines of the dispatch rules: the FP64 Arnoldi step in one
launch or several, the side-by-side FP64 transforms, the RK update's two forms,
the register-tiled training convolutions and the tensor-core row kernel."""
import numpy as np
import pytest

from oracle import sgn_oracle as O
from oracle import unet_oracle as U
from paper_2306_09731_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# half spectra of 40 to 525,312 entries; one launch serves up to 311,296
# (152 blocks of 512 threads with 4 entries each): 262,656 and 263,168 below
# the line, 525,312 above it
@pytest.mark.parametrize("Nx,Ny", [(8, 8), (8, 512), (512, 8), (64, 2048), (1024, 512), (512, 1024), (1024, 1024)])
@pytest.mark.parametrize("graph", [0, 1])
def test_fp64_gmres_solves_to_its_tolerance(Nx, Ny, graph):
    """The residual of the returned sigma, formed by the oracle's operator in
    FP64: the solver stops at a preconditioned relative residual of 1e-12, at
    most sqrt(2) of that without the half spectrum's weights, and the oracle's
    own rounding of M^-1(L sigma) is below 1e-13 of |M^-1 b|."""
    from paper_2306_09731_gb300.sgn import Solver
    Lx, Ly = 0.1 * Nx + 4.0, 0.1 * Ny + 4.0
    st = I.random_state(Nx, Ny, Lx, Ly, seed=Nx + 3 * Ny)
    G = O.Grid(Nx, Ny, Lx, Ly)
    b = O.divergence_rhs(G, st.vx, st.vy)
    s = Solver(Nx, Ny, Lx, Ly, tol=1e-12, restart=20, graph=graph)
    sig, its, rr, conv = s.gmres_solve(dev(st.h), dev(b), dev(np.zeros_like(b)))
    assert conv and rr <= 1e-12
    sig = sig.cpu().numpy()
    ky, kx = np.meshgrid(2 * np.pi * np.fft.fftfreq(Ny, 1.0 / Ny) / Ly, 2 * np.pi * np.arange(Nx // 2 + 1) / Lx,
                         indexing="ij")
    ky[Ny // 2], kx[:, -1] = 0.0, 0.0  # the Nyquist modes have no first derivative
    minv = 1.0 / (3.0 + kx ** 2 + ky ** 2)
    r = minv * np.fft.rfft2(b - O.elliptic_apply(G, st.h, sig))
    assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(minv * np.fft.rfft2(b))
    s.close()


@pytest.mark.parametrize("g", [1.0, 9.81])
@pytest.mark.parametrize("dealias", [0, 1])
@pytest.mark.parametrize("Nx,Ny", [(64, 64), (256, 32)])
def test_rk_update_with_the_linear_part_in_fp64(g, dealias, Nx, Ny):
    """A step with the FP32 right-hand side against the FP64 path: every stage's
    derivative carries FP32 rounding of its transforms, 64 2^-24 of the largest
    field at most, times the largest wavenumber, and the four stages' weights
    add up to dt."""
    from paper_2306_09731_gb300.sgn import Solver
    L, dt = 20.0, 1e-3
    st = I.gaussian_hump(Nx, L, 0.3) if Nx == Ny else I.random_state(Nx, Ny, L, L, seed=5)
    out = []
    for precision in (0, 2):
        s = Solver(Nx, Ny, L, L, g, precision=precision, dealias=dealias)
        f = [dev(st.h), dev(0 * st.h), dev(0 * st.h), dev(0 * st.h)]
        s.rk4_step(*f, dt, 3)
        out.append([a.cpu().numpy() for a in f[:3]])
        s.close()
    size = max(np.linalg.norm(a) for a in out[0])
    bound = 3 * dt * 64 * 2.0 ** -24 * (np.pi * max(Nx, Ny) / L) * g * size
    for a, r in zip(*out):
        assert np.linalg.norm(a - r) <= bound


# odd batches, 16 to 128 columns, channel counts down to the first layer's 4
@pytest.mark.parametrize("n,B,arch", [(64, 3, U.DEFAULT_ARCH), (128, 1, (2, (16, 48))), (16, 5, (2, (48, 16)))])
def test_training_tiles_match_the_oracle(n, B, arch):
    """FP32 sums of at most n^2 B = 16,384 products in a tree over blocks:
    relative error of a gradient below 1e-4, as for the library's other sizes."""
    from paper_2306_09731_gb300.unet import UNet
    rng = np.random.default_rng(n + B)
    p = U.init_params(n, arch).astype(np.float32)
    x = rng.standard_normal((B, 4, n, n)).astype(np.float32)
    t = (0.1 * rng.standard_normal((B, 1, n, n))).astype(np.float32)
    net = UNet(n, max_batch=B, bf16=False, arch=arch)
    net.set_params(dev(p))
    out = net.forward(dev(x)).cpu().numpy()
    loss = net.backward(dev(t))
    g = net.grads().cpu().numpy()
    net.close()
    p64, x64, t64 = (a.astype(np.float64) for a in (p, x, t))
    ro, cache = U.forward(p64, x64, arch)
    rloss, rg = U.backward(p64, ro, cache, t64, arch)
    assert rel(out, ro) < 1e-5
    assert abs(loss - rloss) < 1e-5 * rloss
    assert rel(g, rg) < 1e-4


# (B, H, W, C0, up0, C1, Co): chunk counts that are no multiple of four (48, 80, 112 channels), rows of 2 to
# 1024 pixels, a grid that one tile covers, one that wraps in a single row pair
@pytest.mark.parametrize("B,H,W,C0,up0,C1,Co", [
    (1, 64, 2, 48, 0, 0, 32), (2, 32, 4, 16, 0, 0, 48), (1, 2, 128, 48, 0, 16, 32), (3, 16, 8, 80, 0, 0, 16),
    (1, 4, 512, 16, 1, 0, 16), (1, 16, 64, 112, 0, 0, 32), (1, 2, 64, 32, 0, 48, 96), (1, 2, 1024, 96, 0, 0, 32)])
def test_row_kernel_edges(B, H, W, C0, up0, C1, Co):
    from test_gpu_unet import test_tensor_core_layer_matches_oracle_convolution as check
    check(B, H, W, C0, up0, C1, Co)
