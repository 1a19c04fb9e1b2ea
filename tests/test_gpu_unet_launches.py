"""How many kernels one inference call launches, and what a solver counts for it.

The call is captured and the kernel nodes of the graph are counted; a solver
with the network attached at out_scale 0 takes the same steps as without, plus
per corrected stage (stage 4, and stage 2 after the first step) the two
restriction and two prolongation kernels and one inference.
"""
import ctypes

import numpy as np
import pytest

from paper_2306_09731_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("arch", [(2, (16, 16)), (3, (16, 32, 32))])
def test_launch_count_of_an_inference(arch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_09731_gb300.sgn import Solver
    from paper_2306_09731_gb300.unet import UNet
    n = 32
    net = UNet(n, max_batch=1, bf16=True, seed=1, arch=arch)
    x = torch.zeros((1, 4, n, n), dtype=torch.float32, device="cuda")
    out = net.infer(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        net.infer(x, out)
    cuda = ctypes.CDLL("libcuda.so.1")
    raw = ctypes.c_void_p(g.raw_cuda_graph())
    count = ctypes.c_size_t(0)
    assert cuda.cuGraphGetNodes(raw, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cuda.cuGraphGetNodes(raw, nodes, ctypes.byref(count)) == 0
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    assert kernels == 4 * arch[0] - 2

    st = I.gaussian_hump(64, 20.0, 0.3)
    counts = []
    for attach in (False, True):
        s = Solver(64, 64, 20.0, 20.0, precision=2, guess=2)
        if attach:
            s.set_learned_guess(net, n, out_scale=0.0)
        f = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (st.h, st.vx, st.vy, st.sigma)]
        s.rk4_step(*f, 1e-3, 3)
        counts.append((s.profile()["launches"], s.stats()["matvecs"]))
        s.close()
    net.close()
    assert counts[1][1] == counts[0][1]
    corrected = 5  # of 3 steps
    assert counts[1][0] - counts[0][0] == corrected * (4 + kernels)
