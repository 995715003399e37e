"""Plane sweeps that take more than one round: FP32 digit transforms of more rows than one block of
digits holds (128 per SM), in every layout of their rows, and FP64 mode solves of more than 32 warp
tasks per SM."""
import numpy as np
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import TOL, rel_max_err, rounded, to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

A = (1.0, 0.5, 0.25)


def sweep(lib, u, b, dt, method, omega, n):
    nz, ny, nx = u.shape
    with lib.Context(nx, ny, nz, A, block="plane", method=method, dtype=dt, omega=omega,
                     plane_math="simt") as ctx:
        ut, bt = to_dev(u, dt), to_dev(b, dt)
        ctx.sweep(ut, bt, n)
        assert ctx.last_error() == 0
        return to_np(ut)


@pytest.mark.parametrize("nsweeps", [1, 3])
@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0)])
@pytest.mark.parametrize("shape", [(100, 150, 140), (97, 401, 101), (96, 52, 800)],
                         ids=lambda s: "x".join(map(str, s)))
def test_fp32_digits_in_blocks(brs, shape, method, omega, nsweeps, monkeypatch):  # noqa: F811
    """Each form is within the per-sweep tolerance of the exact sweep."""
    nx, ny, nz = shape
    u = rounded(initial_guess((nz, ny, nx)), "f32")
    b = rounded(rhs((nz, ny, nx)), "f32")
    got = sweep(brs, u, b, "f32", method, omega, nsweeps)
    monkeypatch.setenv("BRSMOOTH_MODE_SLICES", "0")
    ref = sweep(brs, u, b, "f32", method, omega, nsweeps)
    assert np.max(np.abs(got - ref)) <= 2 * nsweeps * TOL["f32"] * np.max(np.abs(u))


@pytest.mark.parametrize("nsweeps", [1, 2])
@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("jacobi", 1.0), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("shape", [(500, 5, 331), (60, 4, 2611)], ids=lambda s: "x".join(map(str, s)))
def test_fp64_modes_in_rounds(brs, orc, shape, method, omega, nsweeps):  # noqa: F811
    """10 444 to 10 592 warp tasks (half of them per colour): two and three rounds of 32 warps on each of
    152 SMs."""
    nx, ny, nz = shape
    u, b = initial_guess((nz, ny, nx)), rhs((nz, ny, nx))
    got = sweep(brs, u, b, "f64", method, omega, nsweeps)
    ref = u
    for _ in range(nsweeps):
        ref = orc.sweep(ref, b, A, block="plane", omega=omega,
                        method="jacobi" if method == "jacobi" else "gs_zebra")
    assert rel_max_err(got, ref) <= nsweeps * TOL["f64"]
