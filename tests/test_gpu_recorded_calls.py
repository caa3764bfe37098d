"""Calls that change what a batch's steps read, recorded into a graph: a replay
writes what was asked for when it was recorded."""
import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_recorded_frame_switch_leaves_a_batch_its_arguments():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    side = torch.cuda.Stream()
    prob = W.periodic_suspension(n=256, count=8, seed=5)
    want, got = (D.Simulation(prob, stream=int(side.cuda_stream)) for _ in range(2))
    for s in (want, got):
        s.step(4)
        s.set_moving_frame(-1)          # allocates the frame's offset
        s.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
        got.set_moving_frame(0)
        got.set_moving_frame(-1)
    junk = [W.periodic_suspension(n=128, count=2, seed=k) for k in range(3)]       # (other frames on this stack)
    with torch.cuda.stream(side):
        graph.replay()
    side.synchronize()
    batch = D.Batch([got, D.Simulation(junk[0], stream=int(side.cuda_stream))])
    batch.step(6)
    want.step(6)
    assert batch.errors() == [D.OK, D.OK]
    assert np.array_equal(want.populations(), got.populations())
    for x, y in zip(want.forces(), got.forces()):
        assert np.array_equal(x, y)
    batch.close()
    for s in (want, got):
        s.close()
