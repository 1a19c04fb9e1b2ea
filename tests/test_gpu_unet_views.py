"""Training on a caller's input that starts at no 16-byte boundary.

A contiguous float32 view may begin at any element of a larger tensor; the
values read are the same, so outputs, loss and gradients are those of an aligned
copy bit for bit, in both tile shapes of the first layer (4 and 8 pixels a
thread) and both activation types.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def cuda_ready():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n,B,arch", [(16, 3, None), (128, 4, (2, (32, 16)))])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_view_equals_its_aligned_copy(n, B, arch, bf16, offset):
    from paper_2306_09731_gb300.unet import UNet
    rng = np.random.default_rng(n + offset)
    size = B * 4 * n * n
    base = torch.tensor(rng.standard_normal(size + 4).astype(np.float32), device="cuda")
    t = torch.tensor(rng.standard_normal((B, 1, n, n)).astype(np.float32), device="cuda")
    view = base[offset:offset + size].view(B, 4, n, n)
    copy = view.clone()
    assert view.is_contiguous() and view.data_ptr() % 16 == 4 * offset and copy.data_ptr() % 16 == 0
    got = []
    for x in (view, copy):
        net = UNet(n, max_batch=B, bf16=bf16, seed=3, arch=arch)
        got.append((net.forward(x), net.backward(t), net.grads(), net.infer(x)))
        net.close()
    assert got[0][1] == got[1][1]
    for i in (0, 2, 3):
        assert torch.equal(got[0][i], got[1][i])
