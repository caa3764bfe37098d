"""The calls a strip shares with a whole lattice: the launch shape, the
autotuner, the sweep's timing.

A strip steps through ``begin`` / ``end``; without an exchange between them
its halo rows and force sums stay its own, which is enough here: the same
strip is compared with itself.
"""
import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D.load_library()
    return torch.cuda.Stream()


def problem(nx=160, ny=96):
    return W.Problem(nx=nx, ny=ny, tau=0.7, eps=2.0, u0=(0.01, -0.004), gravity=(0.0, -2e-5),
                     west=W.Side(W.VELOCITY, 0.01, 0.0), east=W.Side(W.PRESSURE), south=W.wall(), north=W.wall(),
                     wan_turek=W.wan_turek_defaults(5.0, 1.3, 1.0, 2e-5),
                     particles=[W.Particle(20.3, 30.2, 6.0, ux=0.02, uy=0.01, omega=0.002, rho_s=1.3),
                                W.Particle(90.6, 47.4, 5.0, ux=-0.01, uy=0.015, omega=-0.001, rho_s=1.1)])


def steps(s, n):
    for _ in range(n):
        s.begin()
        s.end()


def result(s):
    F, Fc, S = s.forces()
    return s.populations(), F, Fc, S


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_every_shape_gives_a_strip_the_same_bits(stream, storage):
    ref = None
    for shape in [(8, 0), (2, 0), (4, 0), (8, 1), (4, 2), (2, 1)]:
        s = D.Strip(problem(), 0, 48, storage, int(stream.cuda_stream))
        s.set_shape(*shape)
        steps(s, 9)
        got = result(s)
        s.close()
        ref = ref or got
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), shape


def test_a_strip_runs_in_the_shape_that_is_set(stream):
    """One block of two warps on each SM keeps an eighth of the default's row
    segments in flight (two of 5 KB an SM: below 2 TB/s at a microsecond's
    latency), so a strip larger than the L2 takes more than 1.5 times as long."""
    import torch
    s = D.Strip(W.Problem(nx=2048, ny=2048, tau=0.8, eps=2.0), 0, 1024, "fp32", int(stream.cuda_stream))
    ms = {}
    for shape in [(8, 0), (2, 1)]:
        s.set_shape(*shape)
        steps(s, 3)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(stream)
        steps(s, 20)
        b.record(stream)
        b.synchronize()
        ms[shape] = a.elapsed_time(b)
    s.close()
    assert ms[(2, 1)] > 1.5 * ms[(8, 0)], ms


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_autotune_times_the_strips_own_sweep(stream, storage):
    tuned, plain = (D.Strip(problem(nx=176, ny=104), 8, 104, storage, int(stream.cuda_stream)) for _ in range(2))
    steps(tuned, 3)
    before = tuned.launches
    w, b = tuned.autotune(reps=2)
    assert w in (2, 4, 8) and b >= 0
    assert tuned.launches > before
    before = tuned.launches
    assert tuned.autotune(reps=2) == (w, b) and tuned.launches == before     # cached: nothing launched
    steps(tuned, 6)
    steps(plain, 9)
    for x, y in zip(result(tuned), result(plain)):
        assert np.array_equal(x, y)
    tuned.close()
    plain.close()


@pytest.mark.parametrize("method", [W.METHOD_DI, W.METHOD_PS])
def test_timing_records_every_sweep_of_a_strip(stream, method):
    prob = problem()
    prob.method = method
    s = D.Strip(prob, 0, 48, "fp32", int(stream.cuda_stream))
    s.set_timing(True)
    assert s.sweep_time() == (0.0, 0)
    steps(s, 70)                            # past one allotment of events
    ms, n = s.sweep_time()
    assert n == 70 and ms > 0.0
    s.set_timing(False)
    steps(s, 2)
    assert s.sweep_time()[1] == 0
    s.close()
