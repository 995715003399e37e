"""FP64 plane sweeps with the x-transforms by digits on the tensor cores, against the same sweeps
with the products on the FP64 pipe: one-sweep calls (two transforms per sweep) and calls of several
(x-sine form), at row lengths around the digit kernels' tile edges, at their shortest and longest,
ragged ny and nz, and rows of very different magnitudes."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import TOL, rounded, to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(47, 5, 3), (48, 33, 5), (49, 7, 1), (63, 6, 2), (64, 129, 2), (65, 4, 3), (96, 1, 9),
          (127, 3, 4), (128, 16, 9), (255, 5, 2), (256, 40, 3), (257, 3, 3), (333, 6, 5), (479, 4, 2),
          (512, 3, 2), (64, 300, 70)]


def sweep(lib, u, b, method, omega, n):
    nz, ny, nx = u.shape
    with lib.Context(nx, ny, nz, (1.0, 0.5, 0.25), block="plane", method=method, dtype="f64",
                     omega=omega) as ctx:
        ut, bt = to_dev(u, "f64"), to_dev(b, "f64")
        ctx.sweep(ut, bt, n)
        assert ctx.last_error() == 0
        return to_np(ut)


@pytest.mark.parametrize("nsweeps", [1, 3])
@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_digits_equal_fp64_products(brs, shape, method, omega, nsweeps, monkeypatch):  # noqa: F811
    """Both forms round each transform within a few n^(1/2) units of 2^-53 of its row's 2-norm; the
    sweeps contract.  1e-13 is ten times n 2^-53 at n = 512."""
    nx, ny, nz = shape
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    got = sweep(brs, u, b, method, omega, nsweeps)
    monkeypatch.setenv("BRSMOOTH_MODE_SLICES", "0")
    ref = sweep(brs, u, b, method, omega, nsweeps)
    assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(u))


SHAPES32 = [(95, 7, 4), (96, 33, 5), (97, 5, 3), (128, 130, 3), (129, 4, 2), (200, 37, 9), (255, 3, 3),
            (256, 6, 70), (300, 257, 2), (479, 5, 2), (100, 31, 200)]


@pytest.mark.parametrize("nsweeps", [1, 3])
@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("shape", SHAPES32, ids=lambda s: "x".join(map(str, s)))
def test_fp32_digits_equal_products(brs, shape, method, omega, nsweeps, monkeypatch):  # noqa: F811
    """FP32 contexts on CUDA cores: each form is within the per-sweep tolerance of the exact sweep."""
    nx, ny, nz = shape
    u = rounded(initial_guess((nz, ny, nx)), "f32")
    b = rounded(rhs((nz, ny, nx)), "f32")

    def run():
        with brs.Context(nx, ny, nz, (1.0, 0.5, 0.25), block="plane", method=method, dtype="f32",
                         omega=omega, plane_math="simt") as ctx:
            ut, bt = to_dev(u, "f32"), to_dev(b, "f32")
            ctx.sweep(ut, bt, nsweeps)
            assert ctx.last_error() == 0
            return to_np(ut)

    got = run()
    monkeypatch.setenv("BRSMOOTH_MODE_SLICES", "0")
    assert np.max(np.abs(got - run())) <= 2 * nsweeps * TOL["f32"] * np.max(np.abs(u))


@pytest.mark.parametrize("scale", [1e-300, 1e-250, 1.0, 1e250, 1e300])
def test_rows_are_scaled_one_by_one(brs, scale, monkeypatch):  # noqa: F811
    """Planes of magnitudes 1 .. 1e-30 of `scale`, apart enough (az = 1e-200) that each plane keeps
    its own: every plane has its own relative accuracy, at the ends of the range too."""
    nx, ny, nz = 100, 6, 8
    u = initial_guess((nz, ny, nx)) * scale * 10.0 ** (-4.0 * np.arange(nz))[:, None, None]
    b = np.zeros_like(u)

    def run():
        with brs.Context(nx, ny, nz, (1.0, 0.5, 1e-200), block="plane", method="jacobi",
                         dtype="f64") as ctx:
            ut, bt = to_dev(u, "f64"), to_dev(b, "f64")
            ctx.sweep(ut, bt, 3)
            return to_np(ut)

    got = run()
    monkeypatch.setenv("BRSMOOTH_MODE_SLICES", "0")
    ref = run()
    tiny = np.finfo(np.float64).tiny
    for k in range(nz):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-13 * np.max(np.abs(u[k])) + 1e3 * tiny


def test_nan_and_infinity_stay_in_their_rows(brs):  # noqa: F811
    nx, ny, nz = 100, 8, 4
    for bad in (np.nan, np.inf):
        u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
        u[3, 2, 5] = bad
        got = sweep(brs, u, b, "jacobi", 0.8, 1)
        assert not np.isfinite(got[2:]).all() and np.isfinite(got[:2]).all()
        assert not np.isfinite(got[3, 2, 5]) and not np.isfinite(got[2]).any()
