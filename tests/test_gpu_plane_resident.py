"""FP32 plane calls whose mode-line sweeps run on chip (clusters, one mode each) against the
streaming mode sweep, bit for bit: one plane to more planes than one CTA holds, lines of every lane
layout, odd plane counts, more and fewer modes than clusters.  Rows that TMA cannot stage have no
streaming form: they are compared with the per-sweep form, which solves the same planes with two
FP32 transforms per sweep."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import TOL, rel_max_err, rounded, to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

STREAM = [(32, 32, 1, "auto"), (32, 32, 2, "auto"), (64, 32, 33, "auto"), (32, 64, 7, "auto"),
          (96, 128, 21, "auto"), (160, 96, 130, "auto"), (64, 256, 111, "auto"),
          (256, 256, 64, "auto"), (32, 256, 300, "auto"), (32, 384, 75, "auto"), (32, 512, 99, "auto"),
          (700, 64, 5, "simt"), (33, 16, 40, "simt"), (5, 12, 9, "simt"), (3, 4, 260, "simt")]
RAGGED = [(48, 19, 12), (50, 50, 7), (60, 101, 230), (57, 190, 64), (64, 255, 100), (49, 301, 6),
          (48, 509, 57), (200, 7, 3)]


def sweep(lib, u, b, method, omega, n, math):
    nz, ny, nx = u.shape
    with lib.Context(nx, ny, nz, (1.0, 0.5, 0.25), block="plane", method=method, dtype="f32",
                     omega=omega, plane_math=math) as ctx:
        ut, bt = to_dev(u, "f32"), to_dev(b, "f32")
        ctx.sweep(ut, bt, n)
        assert ctx.last_error() == 0
        return to_np(ut)


@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("case", STREAM, ids=lambda c: "x".join(map(str, c)))
def test_resident_equals_streaming(brs, case, method, omega, monkeypatch):  # noqa: F811
    nx, ny, nz, math = case
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    got = sweep(brs, u, b, method, omega, 5, math)
    monkeypatch.setenv("BRSMOOTH_MODE_RESIDENT", "0")
    assert np.array_equal(got, sweep(brs, u, b, method, omega, 5, math))


@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0)])
@pytest.mark.parametrize("shape", RAGGED, ids=lambda s: "x".join(map(str, s)))
def test_ragged_rows(brs, shape, method, omega, monkeypatch):  # noqa: F811
    """Four sweeps: four times the per-sweep FP32 tolerance."""
    nx, ny, nz = shape
    u = rounded(initial_guess((nz, ny, nx)), "f32")
    b = rounded(rhs((nz, ny, nx)), "f32")
    got = sweep(brs, u, b, method, omega, 4, "simt")
    monkeypatch.setenv("BRSMOOTH_PLANE_MODES", "0")
    assert rel_max_err(got, sweep(brs, u, b, method, omega, 4, "simt")) <= 4 * TOL["f32"]
