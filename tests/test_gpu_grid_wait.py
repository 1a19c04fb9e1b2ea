"""The bounded wait of the one-launch FP64 orthogonalisation runs out.

A grid barrier that waits for one block more than the grid has never opens: the
call must end by itself with SGN_ECUDA, the host-driven solve and the step graph
alike, and the handle's next call must give what it gave before
(sgn_grid_wait_selftest). Grids of 1, 2, 130 and 152 blocks, the last with up to four
entries a thread.
"""
import time

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Nx,Ny", [(8, 8), (16, 16), (256, 256), (1024, 512)])
def test_run_out_wait_is_an_error_and_the_handle_goes_on(Nx, Ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_09731_gb300 import sgn as S
    t0 = time.perf_counter()
    assert S.load_library().sgn_grid_wait_selftest(Nx, Ny, torch.cuda.current_stream().cuda_stream) == S.SGN_OK
    assert time.perf_counter() - t0 < 60


def test_other_grids_are_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_09731_gb300 import sgn as S
    lib = S.load_library()
    assert lib.sgn_grid_wait_selftest(1024, 1024, None) == S.SGN_EINVAL
    assert lib.sgn_grid_wait_selftest(24, 8, None) == S.SGN_EINVAL
