"""Lattices without particles, which step by launches of the sweep alone up to
30000 row segments and by fused steps beyond: the same bits as in a batch
(fused), alone, in pieces, timed, tuned and replayed from a graph."""
import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D.load_library()
    return torch


def flow(nx, ny, walls):
    sides = dict(west=W.Side(W.VELOCITY, 0.02, 0.003), east=W.Side(W.PRESSURE), south=W.wall(0.01), north=W.wall(-0.02)) if walls else {}
    return W.Problem(nx=nx, ny=ny, tau=0.7, eps=1.5, u0=(0.01, 0.004), **sides)


def stirred(sim, seed=1):
    """A start that no symmetry keeps uniform."""
    f = sim.populations()
    sim.set_populations(f * (1.0 + 1e-3 * np.random.default_rng(seed).standard_normal(f.shape)))
    return sim


@pytest.mark.parametrize("nx,ny,walls", [(3, 3, True), (257, 5, True), (130, 700, False), (128, 30000, False),
                                         (128, 30001, False), (1100, 1100, True), (2048, 1876, True)])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_same_bits_as_fused_steps(torch, nx, ny, walls, storage):
    side = torch.cuda.Stream()
    a, b, c = (stirred(D.Simulation(flow(nx, ny, walls), storage=storage, stream=int(side.cuda_stream))) for _ in range(3))
    batch = D.Batch([b])
    for n in (1, 8, 5):
        a.step(n)
        batch.step(n)
    batch.sync()
    fa = a.populations()
    assert np.array_equal(fa, b.populations())
    assert all(np.array_equal(x, y) for x, y in zip(a.fields(), b.fields()))
    # timed, tuned, from a graph: 3 + 2 + 2 x 4 + 1 steps
    c.set_timing(True)
    c.step(3)
    ms, n = c.sweep_time()
    assert n == 3 and ms > 0.0
    c.set_timing(False)
    c.autotune(reps=1)
    c.step(2)
    c.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
        c.step(4)
    with torch.cuda.stream(side):
        graph.replay()
        graph.replay()
    side.synchronize()
    c.step(1)
    assert np.array_equal(fa, c.populations())
    assert a.force_mean()[1] == b.force_mean()[1] == c.force_mean()[1] == 14
    batch.close()
    for s in (a, b, c):
        s.close()


@pytest.mark.parametrize("nx,ny", [(130, 70), (2100, 2100)])
def test_ps_without_particles_is_the_plain_flow(torch, nx, ny):
    """No covered cell: the same steps, several to a call (by sweeps, and fused)."""
    side = torch.cuda.Stream()
    prob = flow(nx, ny, True)
    ps = flow(nx, ny, True)
    ps.method = W.METHOD_PS
    a, b = (stirred(D.Simulation(p, stream=int(side.cuda_stream))) for p in (prob, ps))
    for n in (1, 6):
        a.step(n)
        b.step(n)
    assert np.array_equal(a.populations(), b.populations())
    assert all(np.array_equal(x, y) for x, y in zip(a.fields(), b.fields()))
    for s in (a, b):
        s.sync()
        s.close()


def test_on_the_default_streams(torch):
    """The legacy and the per-thread default stream take the same steps."""
    want = stirred(D.Simulation(flow(300, 120, True), stream=int(torch.cuda.Stream().cuda_stream)))
    want.step(9)
    for handle in (0, 1, 2):            # NULL, cudaStreamLegacy, cudaStreamPerThread
        s = stirred(D.Simulation(flow(300, 120, True), stream=handle))
        s.step(9)
        assert np.array_equal(s.populations(), want.populations())
        s.sync()
        s.close()
    want.close()
