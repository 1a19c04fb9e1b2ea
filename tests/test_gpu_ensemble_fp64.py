"""FP64 ensembles: members whose Arnoldi steps orthogonalise in one cooperative
launch each, on their own streams at the same time, get the bits that each gets
alone (sgn_rk4_step_batch against sgn_rk4_step)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# 17 to 152 blocks a launch, and one grid above the one-launch form's line
GRIDS = [(256, 16, 60.0, 15.0), (256, 256, 60.0, 60.0), (512, 256, 120.0, 60.0), (1024, 1024, 60.0, 60.0)]


@pytest.mark.parametrize("graph", [1, 0])
def test_fp64_batch_equals_members_one_by_one(graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_09731_gb300.ensemble import Ensemble, perturbed_members
    states = perturbed_members(9, seed=11, grids=GRIDS)
    a = Ensemble(states, precision=0, guess=2, graph=graph)
    assert a.step(2e-3, 2) == [0] * 9
    b = Ensemble(states, precision=0, guess=2, graph=graph)
    b.step_one_by_one(2e-3, 2)
    torch.cuda.synchronize()
    for fa, fb in zip(a.fields, b.fields):
        for x, y in zip(fa, fb):
            assert torch.equal(x, y)
    for sa, sb in zip(a.solvers, b.solvers):
        assert sa.stats()["matvecs"] == sb.stats()["matvecs"]
    a.close()
    b.close()
