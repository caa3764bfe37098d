"""A lattice stepped alone against the same lattice in a batch, at the sizes
where the way through a step changes: records loaded beside the mask (discs
times segments up to 4096, never in a batch), and with two warps to a segment
or one."""
import numpy as np
import pytest

from paper_2106_08950_gb300 import dilbm as D
from tests.test_gpu_fused import _grid_of_discs, stream  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,count", [(256, 64, 32), (256, 65, 32), (384, 1365, 1), (384, 1366, 1), (512, 512, 2),
                                         (512, 513, 2)])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_records_beside_the_mask(stream, nx, ny, count, storage):  # noqa: F811
    prob = _grid_of_discs(nx, ny, count, True)
    a, b = (D.Simulation(prob, storage=storage, stream=int(stream.cuda_stream)) for _ in range(2))
    batch = D.Batch([b])
    for n in (1, 12, 7):
        a.step(n)
        batch.step(n)
        assert np.array_equal(a.populations(), b.populations())
        assert all(np.array_equal(x, y) for x, y in zip(a.forces(), b.forces()))
    batch.sync()
    batch.close()
    a.close()
    b.close()
