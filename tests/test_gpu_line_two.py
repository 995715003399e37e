"""FP32 x-line Jacobi calls of several sweeps (two sweeps per pass over the grid) against one-sweep
passes, bit for bit: tiles of 14 lines with ragged ends, runs of planes that cross tiles, one plane,
one line, widths that fill and do not fill the lanes, odd sweep counts."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(256, 14, 40), (256, 15, 9), (256, 1, 3), (256, 13, 1), (248, 29, 17), (136, 200, 30),
          (128, 43, 64), (100, 57, 31), (68, 14, 2), (72, 300, 7), (256, 256, 60), (192, 5, 700)]


def sweep(lib, u, b, n, omega):
    nz, ny, nx = u.shape
    with lib.Context(nx, ny, nz, (1.0, 0.5, 0.25), block="line", method="jacobi", dtype="f32",
                     omega=omega) as ctx:
        ut, bt = to_dev(u, "f32"), to_dev(b, "f32")
        ctx.sweep(ut, bt, n)
        assert ctx.last_error() == 0
        return to_np(ut)


@pytest.mark.parametrize("nsweeps,omega", [(3, 0.8), (5, 0.8), (4, 1.0)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_two_sweeps_equal_one_by_one(brs, shape, nsweeps, omega, monkeypatch):  # noqa: F811
    nx, ny, nz = shape
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    monkeypatch.setenv("BRSMOOTH_LINE_TWO", "2")  # also below the size rule
    got = sweep(brs, u, b, nsweeps, omega)
    monkeypatch.setenv("BRSMOOTH_LINE_TWO", "0")
    assert np.array_equal(got, sweep(brs, u, b, nsweeps, omega))
