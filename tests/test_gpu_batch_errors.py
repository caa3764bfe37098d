"""Every member of a batch that failed says so, not the first one alone."""
import pytest

from paper_2106_08950_gb300 import dilbm as D
from paper_2106_08950_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_every_failed_member_is_reported():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stream = int(torch.cuda.Stream().cuda_stream)
    good = W.periodic_suspension(n=128, count=2, seed=1)
    # a fixed disc in a fast flow at tau -> 1/2 goes unstable
    bad = W.cylinder_drag(nx=96, ny=64, r=8.0, cx=30.0, cy=32.0, u=0.5)
    bad.tau = 0.5001
    members = [D.Simulation(p, stream=stream) for p in (good, bad, good, bad, bad)]
    batch = D.Batch(members)
    batch.step(400)
    codes = (D.C.c_int * len(members))()
    D.check(batch.L.dilbm_batch_errors(batch.h, codes))
    assert list(codes) == [D.OK, D.ERR_UNSTABLE, D.OK, D.ERR_UNSTABLE, D.ERR_UNSTABLE]
    with pytest.raises(D.DilbmError) as e:
        batch.sync()
    assert e.value.code == D.ERR_UNSTABLE and "member 1" in str(e.value)
    batch.close()
    for m in members:
        m.close()
