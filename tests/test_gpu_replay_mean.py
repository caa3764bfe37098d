"""The running mean of the forces counts the steps that ran: recorded launches
count as often as they are replayed, and not when they are recorded."""
import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("steps,replays", [(4, 0), (4, 1), (2, 5)])
def test_mean_over_replayed_steps(batched, steps, replays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    probs = [W.periodic_suspension(n=256, count=8, seed=5), W.periodic_suspension(n=192, count=4, seed=6)][: 1 + batched]
    side = torch.cuda.Stream()
    want, got = ([D.Simulation(p, stream=int(side.cuda_stream)) for p in probs] for _ in range(2))
    advance = [(lambda k, b=D.Batch(g): b.step(k)) if batched else g[0].step for g in (want, got)]
    for f in advance:
        f(3)
    for s in want + got:
        s.force_mean_reset()
    advance[0](2 + steps * replays)
    advance[1](2)
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
        advance[1](steps)
    with torch.cuda.stream(side):
        for _ in range(replays):
            graph.replay()
    side.synchronize()
    for a, b in zip(want, got):
        (ma, na), (mb, nb) = a.force_mean(), b.force_mean()
        assert na == nb == 2 + steps * replays
        assert np.array_equal(ma, mb)
        b.force_mean_reset()
        assert b.force_mean()[1] == 0
    advance[1](1)
    assert got[0].force_mean()[1] == 1
    assert np.array_equal(got[0].force_mean()[0], got[0].forces()[0])
    for s in want + got:
        s.close()


def test_mean_of_a_strip_and_without_particles():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stream = int(torch.cuda.Stream().cuda_stream)
    prob = W.Problem(nx=160, ny=96, tau=0.7, eps=2.0, u0=(0.01, 0.0), particles=[W.Particle(20.3, 30.2, 6.0, fixed=True)])
    s = D.Strip(prob, 0, 48, "fp32", stream)
    total = np.zeros(3)
    for k in range(5):
        s.begin()
        s.end()
        if k == 1:
            s.force_mean_reset()
        if k > 1:
            total += s.forces()[0][0]
    m, n = s.force_mean()
    assert n == 3 and np.allclose(m[0], total / 3, rtol=1e-14, atol=0.0)
    s.close()
    s = D.Simulation(W.Problem(nx=64, ny=32, tau=0.8, eps=2.0), stream=stream)
    s.step(7)
    assert s.force_mean()[1] == 7
    s.force_mean_reset()
    s.step(3)
    assert s.force_mean()[1] == 3
    s.close()
