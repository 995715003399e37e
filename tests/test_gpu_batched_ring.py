"""FP32 patch sweeps through the shared-memory ring (patch rows of whole 16-byte pieces) against
the kernel that loads its rows directly, bit for bit: lines of 4 to 32 lanes filled and not, fewer
lines than a warp takes and ragged last groups, one plane, chunks of planes shorter and longer than
the ring and a remainder; plain patches and a level (ghost rows on every face, patches of one line
group and of several)."""
import numpy as np
import pytest

from brs_inputs import batched_fields, uniform_field
from gpu_common import to_dev, to_np
from test_gpu_batched import brs  # noqa: F401
from test_gpu_level import tiling

pytestmark = pytest.mark.gpu

PLAIN = [(nx, ny, nz) for nx, ny, nz in zip((4, 8, 16, 20, 28, 32, 36, 60, 64, 68, 100, 128),
                                            (1, 9, 16, 3, 8, 2, 5, 7, 2, 1, 3, 2),
                                            (33, 1, 5, 6, 4, 17, 2, 9, 40, 8, 3, 5))]
LEVELS = [((2, 2, 2), (16, 9, 5)), ((1, 3, 2), (36, 5, 9)), ((2, 1, 3), (72, 3, 4)),
          ((3, 2, 1), (20, 8, 33))]


def sweep(lib, dims, nbr, u, b, nsweeps):
    with lib.BatchedContext(dims, (1.0, 0.5, 0.25), method="jacobi", dtype="f32", nbr=nbr) as c:
        ut, bt = to_dev(u, "f32"), to_dev(b, "f32")
        c.sweep(ut, bt, nsweeps)
        assert lib.brsmooth_last_error(c.h) == 0
        return to_np(ut)


@pytest.mark.parametrize("kc", [1, 3, 4, 5, 8, 32])
@pytest.mark.parametrize("level", [None, *LEVELS], ids=str)
def test_ring_equals_direct_loads(brs, level, kc, monkeypatch):  # noqa: F811
    dims, nbr = tiling(*level) if level else (np.array(PLAIN), None)
    n = int(np.prod(dims, axis=1).sum())
    u, b = uniform_field((n,), 3), batched_fields(dims, 4, scale_h2=True, h=1 / 33)
    monkeypatch.setenv("BRSMOOTH_BATCH_NOTUNE", "1")
    monkeypatch.setenv("BRSMOOTH_BATCH_KC", str(kc))
    got = sweep(brs, dims, nbr, u, b, 3)
    monkeypatch.setenv("BRSMOOTH_BATCH_ASYNC", "0")
    assert np.array_equal(got, sweep(brs, dims, nbr, u, b, 3))
