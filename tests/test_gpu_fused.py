"""Fused steps: several steps in one launch, particles updated by blocks of
their own while the others sweep.

Each case is stepped in one call and compared bit for bit with the same
lattice stepped one step per call, and with the FP64 oracle: more particles
than a particle warp watches at once, several particles per warp, the smallest
walled lattices (every row an edge row), discs across both periodic edges, a
particle that leaves the lattice with the moving frame, and launches recorded
into a CUDA graph by the caller.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W
from tests import parity as PAR

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D.load_library()
    return torch.cuda.Stream()


def many_small_discs(n=512, per_row=36):
    """per_row^2 small discs on a jittered grid, some in contact range."""
    rng = np.random.default_rng(11)
    h = n / per_row
    parts = [W.Particle((i + 0.5) * h + rng.uniform(-2, 2), (j + 0.5) * h + rng.uniform(-2, 2), 4.0,
                        ux=rng.uniform(-0.01, 0.01), uy=rng.uniform(-0.01, 0.01), rho_s=1.3)
             for i in range(per_row) for j in range(per_row)]
    return W.Problem(nx=n, ny=n, tau=0.8, eps=1.0, gravity=(0.0, -1e-5),
                     wan_turek=W.wan_turek_defaults(4.0, 1.3, 1.0, 1e-5), particles=parts, name="many")


def tiny_walls(nx, ny):
    return W.Problem(nx=nx, ny=ny, tau=0.7, eps=1.5, west=W.Side(W.VELOCITY, 0.01, 0.002), east=W.Side(W.PRESSURE),
                     south=W.wall(0.004), north=W.wall(-0.003), u0=(0.01, 0.0), name=f"walls {nx}x{ny}")


CASES = {
    # 1296 particles; with 2 warps per block and 1 block per SM, 15 particle
    # blocks: 30 warps, 44 particles each (32 watched at a time)
    "many": (many_small_discs, (2, 1), 8),
    "corners": (lambda: W.Problem(nx=130, ny=37, tau=0.8, eps=2.0, wan_turek=W.wan_turek_defaults(5.0, 1.3, 1.0, 1e-5),
                                  particles=[W.Particle(0.4, 36.6, 5.0, ux=-0.02, uy=0.02, rho_s=1.3),
                                             W.Particle(65.0, 12.0, 4.0, omega=0.002, fixed=True)]), (4, 0), 61),
    "walls 3x3": (lambda: tiny_walls(3, 3), (4, 0), 30),
    "walls 129x3": (lambda: tiny_walls(129, 3), (8, 0), 30),
    "walls 257x4": (lambda: tiny_walls(257, 4), (2, 0), 30),
}


@pytest.mark.parametrize("name", CASES)
def test_one_launch_matches_single_steps_and_the_oracle(stream, name):
    make, shape, steps = CASES[name]
    prob = make()
    a, b = (D.Simulation(prob, stream=int(stream.cuda_stream)) for _ in range(2))
    a.set_shape(*shape)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    fa, fb = a.fields(), b.fields()
    assert np.array_equal(a.populations(), b.populations())
    o = O.OracleSim(prob, phi_cutoff=PAR.oracle_cutoff(prob))
    o.step(steps - 1)
    pre = PAR.oracle_pre(o) if prob.particles else None
    o.step(1)
    ok, errs = PAR.compare_fields(fa, o.fields())
    assert ok, errs
    if prob.particles:
        Fa, Ca, Sa = a.forces()
        Fb, Cb, Sb = b.forces()
        assert np.array_equal(Fa, Fb) and np.array_equal(Ca, Cb) and np.array_equal(Sa, Sb)
        Fo, _, So = o.forces()
        ok, e = PAR.compare_forces_terms(Fa, Fo, PAR.force_term_scales(prob, *pre))
        assert ok, e
        ok, e = PAR.compare_state(Sa, So)
        assert ok, e
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_default_stream_and_captured_launches(stream, storage):
    """On the legacy default stream, and replayed from a graph the caller
    captured (an even number of steps, so that a replay starts where it
    ended), the steps are the ones of an ordinary stream."""
    import torch
    prob = W.periodic_suspension(n=256, count=8, seed=5)
    ref = D.Simulation(prob, storage=storage, stream=int(stream.cuda_stream))
    ref.step(18)
    plain = D.Simulation(prob, storage=storage, stream=0)
    plain.step(18)
    side = torch.cuda.Stream()
    cap = D.Simulation(prob, storage=storage, stream=int(side.cuda_stream))
    cap.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
        cap.step(6)
    with torch.cuda.stream(side):
        for _ in range(3):
            graph.replay()
    side.synchronize()
    for sim in (plain, cap):
        assert np.array_equal(sim.populations(), ref.populations())
        for x, y in zip(sim.forces(), ref.forces()):
            assert np.array_equal(x, y)
        sim.close()
    ref.close()


def test_particle_that_leaves_the_lattice(stream):
    """The frame follows one disc; another is carried out of the lattice, where
    no tile holds it: it keeps its update (no force, its velocity)."""
    side = W.Side(W.PRESSURE, 0.0, 0.0, 1.0)
    prob = W.Problem(nx=96, ny=48, tau=0.8, eps=1.5, west=side, east=side, south=W.wall(), north=W.wall(),
                     wan_turek=W.wan_turek_defaults(4.0, 1.2, 1.0, 1e-5),
                     particles=[W.Particle(60.0, 30.0, 4.0, ux=0.2, rho_s=1e4),
                                W.Particle(8.0, 14.0, 4.0, ux=0.0, rho_s=1e4)])
    a, b = (D.Simulation(prob, stream=int(stream.cuda_stream)) for _ in range(2))
    for s in (a, b):
        s.set_moving_frame(0)
    a.step(120)
    for _ in range(120):
        b.step(1)
    Fa, _, Sa = a.forces()
    Fb, _, Sb = b.forces()
    assert a.frame_offset() == b.frame_offset() > 18
    assert Sa[1, 0] < -(4.0 + 4 * prob.eps) and np.array_equal(Fa[1], np.zeros(3))
    assert np.array_equal(Sa, Sb) and np.array_equal(Fa, Fb)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()


@pytest.mark.parametrize("steps,replays", [(2, 1), (2, 5), (4, 3), (8, 2)])
@pytest.mark.parametrize("batched", [False, True])
def test_captured_steps_replay_from_any_step(stream, steps, replays, batched):
    """A recorded even number of steps goes on from wherever the lattice
    stands: after steps taken outside the graph, and by an upload and more
    steps after the replays."""
    import torch
    probs = [W.periodic_suspension(n=256, count=8, seed=5), W.periodic_suspension(n=192, count=4, seed=6)]
    side = torch.cuda.Stream()
    want, got = ([D.Simulation(p, stream=int(s.cuda_stream)) for p in probs[: 1 + batched]] for s in (stream, side))
    advance = [(lambda k, b=D.Batch(g): b.step(k)) if batched else g[0].step for g in (want, got)]
    advance[0](2 + steps * replays)
    advance[1](2)
    for s in got:
        s.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
        advance[1](steps)
    with torch.cuda.stream(side):
        for _ in range(replays):
            graph.replay()
    side.synchronize()
    for after in range(2):
        for a, b in zip(want, got):
            assert np.array_equal(a.populations(), b.populations())
            for x, y in zip(a.forces(), b.forces()):
                assert np.array_equal(x, y)
        for a, b, p in zip(want, got, probs):
            a.set_particles(p.particles)
            b.set_particles(p.particles)
        for f in advance:
            f(5)
    for s in want + got:
        s.close()


def _grid_of_discs(nx, ny, count, walls):
    """`count` small moving discs on a grid, some across tile edges."""
    rows = max(1, int(np.sqrt(count * ny / nx)))
    cols = -(-count // rows)
    rng = np.random.default_rng(7)
    parts = [W.Particle((k % cols + 0.5) * nx / cols, (k // cols + 0.5) * ny / rows, 5.0, ux=rng.uniform(-0.02, 0.02),
                        uy=rng.uniform(-0.02, 0.02), omega=rng.uniform(-1e-3, 1e-3), rho_s=1.3) for k in range(count)]
    sides = dict(west=W.Side(W.VELOCITY, 0.01, 0.0), east=W.Side(W.PRESSURE), south=W.wall(), north=W.wall(0.002)) if walls else {}
    return W.Problem(nx=nx, ny=ny, tau=0.8, eps=1.5, gravity=(0.0, -1e-6), u0=(0.01, 0.0),
                     wan_turek=W.wan_turek_defaults(5.0, 1.3, 1.0, 1e-5), particles=parts, **sides)


# Where a lattice stepped alone takes another way than in a batch: two warps to
# a segment (up to 1518 segments in FP32, 1822 in FP16, on 152 SMs), records
# loaded beside the mask (discs times segments up to 65536), slots by number (up
# to 32 discs), and steps from the end (two buffers over 96 MB).
ALONE = [(256, 759, 2, True, "fp32"), (256, 760, 2, True, "fp32"), (200, 759, 3, False, "fp32"),
         (190, 911, 2, True, "fp16"), (190, 912, 2, True, "fp16"), (3, 5, 0, True, "fp32"), (129, 8, 1, False, "bf16"),
         (512, 512, 32, False, "fp32"), (512, 513, 32, False, "fp32"), (384, 300, 33, True, "fp32"),
         (1184, 1184, 40, False, "fp32"), (1184, 1180, 40, False, "fp32"), (1700, 1700, 8, True, "fp16")]


@pytest.mark.parametrize("nx,ny,count,walls,storage", ALONE)
def test_alone_as_in_a_batch(stream, nx, ny, count, walls, storage):
    prob = _grid_of_discs(nx, ny, count, walls)
    a, b = (D.Simulation(prob, storage=storage, stream=int(stream.cuda_stream)) for _ in range(2))
    batch = D.Batch([b])
    for n in (1, 12, 7):
        a.step(n)
        batch.step(n)
        assert np.array_equal(a.populations(), b.populations())
        assert all(np.array_equal(x, y) for x, y in zip(a.fields(), b.fields()))
        assert all(np.array_equal(x, y) for x, y in zip(a.forces(), b.forces()))
    batch.sync()
    batch.close()
    a.close()
    b.close()


@pytest.mark.parametrize("count", [1, 32, 33])
def test_uploads_in_a_row(stream, count):
    """Uploads between steps, one or several in a row, leave the same state."""
    prob = _grid_of_discs(400, 300, count, True)
    a, b = (D.Simulation(prob, stream=int(stream.cuda_stream)) for _ in range(2))
    moved = [W.Particle(q.x + 1.25, q.y - 0.5, q.r, ux=-q.ux, uy=q.uy, rho_s=1.2, fixed=k % 5 == 0)
             for k, q in enumerate(prob.particles)]
    for times in (1, 3, 2):
        for s, m in ((a, 1), (b, times)):
            s.step(2)
            for k in range(m):
                s.set_particles(prob.particles if k + 1 < m else moved)
            s.step(4)
        assert np.array_equal(a.populations(), b.populations())
        assert all(np.array_equal(x, y) for x, y in zip(a.forces(), b.forces()))
        assert all(np.array_equal(x, y) for x, y in zip(a.fields(), b.fields()))
    a.close()
    b.close()
