"""A batch counts the kernels it launches: fused steps are one launch per group
of members, however many steps a call asks for."""
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members,groups", [(3, 1), (84, 1), (85, 2)])
def test_kernels_of_fused_steps(members, groups):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stream = int(torch.cuda.Stream().cuda_stream)
    sims = [D.Simulation(W.Problem(nx=64, ny=32, tau=0.8, eps=2.0, particles=[W.Particle(20.0, 16.0, 5.0, rho_s=1.2)]),
                         stream=stream) for _ in range(members)]
    batch = D.Batch(sims)
    batch.step(7)
    batch.step(4)
    assert batch.kernels == 2 * groups
    batch.sync()
    assert batch.kernels == 2 * groups + 1          # the error gather
    batch.set_timing(True)
    batch.step(5)
    assert batch.kernels == 7 * groups + 1
    batch.close()
    for s in sims:
        s.close()
