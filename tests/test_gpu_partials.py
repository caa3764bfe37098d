"""Force partials by slot (more than 64 particles, and more than tiles): against the oracle and single steps, with uploads, moving discs over
tile edges and partial last tiles, in a batch, in PS, and in two strips."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as O
from paper_2106_08950_gb300 import build as B
from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W
from tests import parity as PAR
from tests.test_gpu_fused import _grid_of_discs


@pytest.fixture(scope="module")
def stream():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    D.load_library()
    return torch.cuda.Stream()


def test_memory_of_many_small_discs():
    """A particle takes its share of the lists and its state; the partials of
    all of them no more than MAXC (32) slots of 8 rows of 16 bytes a tile."""
    B.build()
    lib = D.load_library()

    def footprint(np_):
        g = D.make_grid(W.Problem(nx=4096, ny=4096, tau=0.8, eps=1.0), "fp32")
        b = C.c_ulonglong()
        assert lib.dilbm_footprint(C.byref(g), np_, C.byref(b)) == D.OK
        return b.value
    tiles = 32 * 512
    assert footprint(84000) - footprint(1) <= tiles * 32 * 8 * 16 + 84000 * 1300
    # few particles: 16 KB each, found by the particle
    assert footprint(64) - footprint(1) == 63 * (128 * 8 * 16 + 15 * 8 + 5 * 4 + 4 + 8 * 8 + 2 * 130 * 4)


def discs(nx, ny, count, r=3.0, **kw):
    prob = _grid_of_discs(nx, ny, count, kw.pop("walls", True))
    for q in prob.particles:
        q.r = r
    prob.eps = 1.0
    for k, v in kw.items():
        setattr(prob, k, v)
    return prob


CASES = {"64 discs, 50 tiles": (lambda: discs(200, 200, 64), 9), "65 discs, 50 tiles": (lambda: discs(200, 200, 65), 9),
         "114 discs, 114 tiles": (lambda: discs(384, 300, 114), 9), "115 discs, 114 tiles": (lambda: discs(384, 300, 115), 9),
         "400 discs": (lambda: discs(520, 261, 400, walls=False), 9),
         "ps": (lambda: discs(300, 203, 90, method=W.METHOD_PS), 5)}


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_against_single_steps_and_the_oracle(stream, name):
    make, steps = CASES[name]
    prob = make()
    a, b, c = (D.Simulation(prob, stream=int(stream.cuda_stream)) for _ in range(3))
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    runs = [a, b]
    if prob.method == W.METHOD_DI:
        batch = D.Batch([c])
        batch.step(steps)
        batch.sync()
        runs.append(c)
    Fa, Ca, Sa = a.forces()
    for s in runs[1:]:
        assert np.array_equal(a.populations(), s.populations())
        assert all(np.array_equal(x, y) for x, y in zip((Fa, Ca, Sa), s.forces()))
    o = O.OracleSim(prob, phi_cutoff=PAR.oracle_cutoff(prob))
    o.step(steps - 1)
    pre = PAR.oracle_pre(o)
    o.step(1)
    ok, errs = PAR.compare_fields(a.fields(), o.fields())
    assert ok, errs
    Fo, _, So = o.forces()
    ok, e = PAR.compare_forces_terms(Fa, Fo, PAR.force_term_scales(prob, *pre))
    assert ok, e
    ok, e = PAR.compare_state(Sa, So)
    assert ok, e
    # uploads, several in a row, between steps
    for s, times in zip(runs, (1, 3, 2)):
        for _ in range(times):
            s.set_particles(prob.particles)
        s.step(4)
    for s in runs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(a.forces(), s.forces()))
    for s in (a, b, c):
        s.close()


@pytest.mark.gpu
def test_two_strips_match_the_whole_lattice(stream):
    """Both strips in one process, exchanged by device copies: the sums are
    added in another order, so the bound is the strips' 1e-6."""
    import torch
    from paper_2106_08950_gb300.strips import device_bytes
    prob = discs(160, 96, 110, walls=False)
    whole = D.Simulation(prob, stream=int(stream.cuda_stream))
    pair = [D.Strip(prob, 0, 48, stream=int(stream.cuda_stream)), D.Strip(prob, 48, 96, stream=int(stream.cuda_stream))]
    buf = []
    for s in pair:
        fpart, ss, sn, rs, rn, n = s.buffers()
        buf.append([device_bytes(fpart, 8 * 5 * len(prob.particles)).view(torch.float64)]
                   + [device_bytes(q, 4 * n) for q in (ss, sn, rs, rn)])
    steps = 40
    whole.step(steps)
    with torch.cuda.stream(stream):
        for _ in range(steps):
            for s in pair:
                s.begin()
            total = buf[0][0] + buf[1][0]
            for k in range(2):
                other = buf[1 - k]
                buf[k][0].copy_(total)
                buf[k][3].copy_(other[2])       # the row south of it: the other's north row
                buf[k][4].copy_(other[1])
            for s in pair:
                s.end()
    F, _, S = whole.forces()
    for s in pair:
        Fs, _, Ss = s.forces()
        assert np.abs(Fs[:, :2] - F[:, :2]).max() <= 1e-6 * np.abs(F[:, :2]).max()
        assert np.abs(Ss[:, :2] - S[:, :2]).max() <= 1e-6
    for s in pair + [whole]:
        s.close()
