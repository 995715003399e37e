"""FP64 x-line sweeps on the caller's layout in several waves of CTAs, with many lines per SM, where a
call of several sweeps takes the line-major form: one-sweep calls, which never do (a call needs two
sweeps at least), against one line-major call, bit for bit."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from test_gpu_box import brs  # noqa: F401
from test_gpu_line_tile import sweep

pytestmark = pytest.mark.gpu

# 438 to 1184 lines per SM: full, ragged and short chunks of 32 cells, even and odd ny and nz
SHAPES = [(32, 300, 222), (41, 401, 300), (63, 333, 271), (16, 450, 400), (96, 260, 257), (1, 400, 250)]


@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("jacobi", 1.0), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_one_sweep_calls_equal_line_major(brs, shape, method, omega, monkeypatch):  # noqa: F811
    nx, ny, nz = shape
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    tile = sweep(brs, u, b, method, omega, [1] * 5)
    monkeypatch.setenv("BRSMOOTH_LINE_SEQ", "2")  # line-major from four sweeps on, on any grid
    assert np.array_equal(tile, sweep(brs, u, b, method, omega, [5]))
