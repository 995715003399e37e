"""FP64 x-line sweeps on the caller's layout against the line-major form: the same operations in
the same order, so the iterates agree bit for bit, whatever the task shape, the calls' length
(b scaled once or per sweep) and the colour rows (odd and even ny and nz)."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(1, 5, 3), (2, 1, 1), (3, 4, 5), (17, 16, 1), (32, 32, 32), (33, 17, 9), (64, 1, 70),
          (127, 31, 3), (256, 9, 6), (384, 33, 20), (511, 6, 5), (512, 24, 17), (40, 100, 101),
          (16, 300, 200), (300, 61, 43)]


def sweep(lib, u, b, method, omega, calls):
    nz, ny, nx = u.shape
    with lib.Context(nx, ny, nz, (1.0, 0.5, 0.25), block="line", method=method, dtype="f64",
                     omega=omega) as ctx:
        ut, bt = to_dev(u, "f64"), to_dev(b, "f64")
        for n in calls:
            ctx.sweep(ut, bt, n)
        assert ctx.last_error() == 0
        return to_np(ut)


@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("jacobi", 1.0), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_tile_equals_line_major(brs, shape, method, omega, monkeypatch):  # noqa: F811
    nx, ny, nz = shape
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    one = sweep(brs, u, b, method, omega, [60])          # long call: b scaled once
    many = sweep(brs, u, b, method, omega, [3] * 20)     # short calls: b scaled per sweep
    monkeypatch.setenv("BRSMOOTH_LINE_SEQ", "2")
    major = sweep(brs, u, b, method, omega, [60])
    assert np.array_equal(one, major) and np.array_equal(many, major)
