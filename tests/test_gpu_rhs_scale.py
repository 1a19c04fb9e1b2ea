"""Elliptic solves and steps whose right-hand side is very small or very large.

L is linear: a right-hand side times 2^k gives sigma times 2^k, as far as FP64
holds the squares of the spectra (1e-154 to 1e154). Both solves stop at a
preconditioned relative residual of 1e-10, sqrt(2) of that without the half
spectrum's weights. M^-1 L has its spectrum between the least and the largest of
1/h and 1/h^3, here h in [0.7, 1.3]: a condition of at most (1.3/0.7)^3 = 6.4, so
the two differ by at most 2 sqrt(2) 6.4 1e-10 = 1.8e-9 relative. On these grids the
norm of the spectrum is up to 128 x 64 / 2 = 4096 times the field's.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
BOUND = 1.8e-9


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.tensor(np.ascontiguousarray(a), device="cuda")


def fields(Nx, Ny):
    y, x = np.mgrid[0:Ny, 0:Nx]
    X, Y = 2 * np.pi * x / Nx, 2 * np.pi * y / Ny
    return 1.0 + 0.2 * np.cos(X) + 0.1 * np.sin(Y + X), np.sin(X) * np.cos(2 * Y) + 0.3 * np.cos(3 * X)


# one launch per orthogonalisation, and (1024 x 1024) several
@pytest.mark.parametrize("Nx,Ny", [(16, 8), (128, 64), (1024, 1024)])
@pytest.mark.parametrize("k", [-495, -480, -301, -299, 299, 301, 480])
def test_solution_scales_with_the_right_hand_side(Nx, Ny, k):
    from paper_2306_09731_gb300.sgn import Solver
    h, b = fields(Nx, Ny)
    s = Solver(Nx, Ny, 20.0, 15.0)
    ref, its0, _, conv0 = s.gmres_solve(dev(h), dev(b))
    sig, its, _, conv = s.gmres_solve(dev(h), dev(b * 2.0 ** k))
    s.close()
    assert conv0 and conv and its <= its0 + 1
    ref, sig = ref.cpu().numpy(), sig.cpu().numpy() * 2.0 ** -k
    assert np.linalg.norm(sig - ref) <= BOUND * np.linalg.norm(ref)


@pytest.mark.parametrize("graph", [0, 1])
def test_steps_of_a_velocity_of_1e_minus_150(graph):
    """Without gravity a small velocity stays small: the step is linear in it, and
    every stage solves for a sigma of its size."""
    from paper_2306_09731_gb300.sgn import Solver
    h, b = fields(128, 64)
    out = []
    for scale in (2.0 ** -100, 2.0 ** -497):
        s = Solver(128, 64, 20.0, 15.0, 0.0, graph=graph)
        f = [dev(h), dev(b * scale), dev(0 * b), dev(0 * b)]
        s.rk4_step(*f, 1e-3, 2)
        st = s.stats()
        s.close()
        assert st["solves"] == 8 and 3 < st["max_iters"] < 60
        out.append([a.cpu().numpy() / (1.0 if i == 0 else scale) for i, a in enumerate(f)])
    for o in out:  # h takes part in no sum of its size: a transform and back
        assert np.linalg.norm(o[0] - h) <= 1e-14 * np.linalg.norm(h)
    for a, r in zip(out[1][1:], out[0][1:]):
        assert np.linalg.norm(a - r) <= 4 * BOUND * np.linalg.norm(out[0][3])
