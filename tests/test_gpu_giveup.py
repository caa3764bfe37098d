"""What a step does when one of its waits runs out, without a fault.

``stall_probe`` makes a particle's update wait for partial sums that no sweep
writes, or the blocks of a launch for one block more than there is.  Every wait
is bounded by 1 s: the status comes back, every lattice that missed steps
reports it, and no later launch waits for it again.
"""
import time

import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W
from tests.test_gpu_fused import many_small_discs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D.load_library()
    return torch.cuda.Stream()


def timed(f):
    t = time.monotonic()
    f()
    return time.monotonic() - t


def sync_code(sim):
    with pytest.raises(D.DilbmError) as e:
        sim.sync()
    return e.value.code


def disc(n, seed):
    return W.periodic_suspension(n=n, count=6, seed=seed)


def same(a, b):
    assert np.array_equal(a.populations(), b.populations())
    for x, y in zip(a.forces(), b.forces()):
        assert np.array_equal(x, y)


# a warp to each particle; counted partials, several particles to a warp; PS:
# one step to a launch; the frame follows the particle that is late
CASES = {"own warps": (lambda: disc(256, 3), None), "counted": (many_small_discs, (2, 1)),
         "ps": (lambda: disc(256, 4), None), "frame": (lambda: disc(192, 5), None)}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("before", [0, 3])
def test_late_partials_are_reported_and_not_waited_for_again(stream, name, before):
    make, shape = CASES[name]
    prob = make()
    if name == "ps":
        prob.method = W.METHOD_PS
    s = D.Simulation(prob, stream=int(stream.cuda_stream))
    if shape:
        s.set_shape(*shape)
    if name == "frame":
        s.set_moving_frame(1)
    s.step(before)
    s.sync()
    s.stall_probe(1)

    def run(n):
        s.step(n)
        assert sync_code(s) == D.ERR_TIMEOUT
    assert 1.0 <= timed(lambda: run(5)) < 2.9           # a wait of 1 s, and the other blocks' for it
    assert timed(lambda: run(300)) < 0.9                # launches after it: none
    assert np.isfinite(s.populations()).all()
    s.close()
    # the device goes on working
    a, b = (D.Simulation(disc(200, 9), stream=int(stream.cuda_stream)) for _ in range(2))
    a.step(4)
    for _ in range(4):
        b.step(1)
    a.sync()
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("late", [0, 1, 2])
def test_a_late_member_ends_the_launch_for_every_lattice_in_it(stream, late):
    probs = [disc(256, 1), many_small_discs(256, 18), disc(320, 2)]
    members = [D.Simulation(p, stream=int(stream.cuda_stream)) for p in probs]
    batch = D.Batch(members)
    batch.step(3)
    members[late].stall_probe(2)
    batch.step(6)
    assert 1.0 <= timed(lambda: batch.errors()) < 2.9
    assert batch.errors() == [D.ERR_TIMEOUT] * 3
    assert timed(lambda: (batch.step(40), batch.errors())) < 0.9
    assert batch.errors() == [D.ERR_TIMEOUT] * 3
    batch.close()
    # beside lattices that are well, one known to have given up is left out
    probs = [disc(256, 7), disc(192, 8)]
    alone, well = ([D.Simulation(p, stream=int(stream.cuda_stream)) for p in probs] for _ in range(2))
    batch = D.Batch([members[late], well[0], members[(late + 1) % 3], well[1]])
    batch.step(9)
    assert batch.errors() == [D.ERR_TIMEOUT, D.OK, D.ERR_TIMEOUT, D.OK]
    for a, m in zip(alone, well):
        a.step(9)
        same(a, m)
    batch.close()
    for s in members + alone + well:
        s.close()


def test_an_abandoned_launch_is_reported_by_every_lattice_in_it(stream):
    probs = [disc(256, 1), disc(192, 2), disc(160, 3)]
    members = [D.Simulation(p, stream=int(stream.cuda_stream)) for p in probs]
    batch = D.Batch(members)
    batch.step(2)
    assert batch.errors() == [D.OK] * 3
    batch.stall_probe()
    assert 1.0 <= timed(lambda: (batch.step(6), batch.errors())) < 2.9
    assert batch.errors() == [D.ERR_TIMEOUT] * 3
    assert timed(lambda: (batch.step(60), batch.errors())) < 0.9
    batch.close()
    for s in members:
        s.close()
    # one lattice, its first steps given up: the copies of the other parity were never written
    s = D.Simulation(probs[0], stream=int(stream.cuda_stream))
    s.set_moving_frame(0)
    s.stall_probe(-1)
    s.step(7)
    assert sync_code(s) == D.ERR_TIMEOUT
    assert timed(lambda: (s.step(51), sync_code(s))) < 0.9
    assert sync_code(s) == D.ERR_TIMEOUT
    s.close()


def test_stall_probe_refusals(stream):
    s = D.Simulation(disc(128, 1), stream=int(stream.cuda_stream))
    for p in (-2, 6):
        with pytest.raises(D.DilbmError):
            s.stall_probe(p)
    s.sync()
    s.close()
    t = D.Strip(W.Problem(nx=64, ny=32, tau=0.8, eps=2.0), 0, 16, stream=int(stream.cuda_stream))
    with pytest.raises(D.DilbmError):
        t.stall_probe(-1)
    t.close()
