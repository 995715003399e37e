"""Plane sweeps of rows whose cells span many orders of magnitude: the digit transforms hold a row as
fixed-point numbers under its largest cell.  Against extended precision they are no further off than
the products in the element type, in the 2-norm, for one spike in a row of small cells, for cells that
decay along the row, and for cells of random exponents."""
import numpy as np
import pytest

from gpu_common import rounded, to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD(4) * np.arctan(LD(1))
A = (1.0, 0.5, 0.25)


def basis(n):
    i = np.arange(1, n + 1)
    return np.sqrt(LD(2) / (n + 1)) * np.sin(np.outer(i, i) % (2 * (n + 1)) * PI / (n + 1))


def exact(u, b, omega, sweeps):
    """Plane Jacobi sweeps in extended precision."""
    u, b, a = u.astype(LD), b.astype(LD), [LD(v) for v in A]
    nz, ny, nx = u.shape
    Sx, Sy = basis(nx), basis(ny)
    eig = [4 * np.sin(np.arange(1, n + 1) * PI / (2 * (n + 1))) ** 2 for n in (nx, ny)]
    lam = a[0] * eig[0][None, :] + a[1] * eig[1][:, None] + 2 * a[2]
    for _ in range(sweeps):
        r = b.copy()
        r[1:] += a[2] * u[:-1]
        r[:-1] += a[2] * u[1:]
        t = np.einsum("yq,zqx->zyx", Sy, r @ Sx) / lam
        u = (1 - LD(omega)) * u + LD(omega) * (np.einsum("yq,zqx->zyx", Sy, t) @ Sx)
    return u


def cells(kind, shape, seed, decades):
    rng = np.random.default_rng(seed)
    v = rng.uniform(-1, 1, shape)
    if kind == "spike":
        v *= 10.0 ** -decades
        v[..., shape[2] // 3] = rng.uniform(0.5, 1, shape[:2])
    elif kind == "decay":
        v *= 10.0 ** (-decades * np.arange(shape[2]) / shape[2])
    else:
        v *= 10.0 ** rng.uniform(-decades, 0, shape)
    return v


@pytest.mark.parametrize("nsweeps", [1, 3])
@pytest.mark.parametrize("decades", [3, 8, 30])
@pytest.mark.parametrize("kind", ["spike", "decay", "random"])
@pytest.mark.parametrize("dt", ["f64", "f32"])
def test_no_further_than_products(brs, dt, kind, decades, nsweeps, monkeypatch):  # noqa: F811
    nx, ny, nz = 130, 9, 6
    u = rounded(cells(kind, (nz, ny, nx), 1, decades), dt)
    b = rounded(cells(kind, (nz, ny, nx), 2, decades), dt)
    ref = exact(u, b, 0.8, nsweeps)

    def distance():
        with brs.Context(nx, ny, nz, A, block="plane", method="jacobi", dtype=dt, omega=0.8,
                         plane_math="simt") as ctx:
            ut, bt = to_dev(u, dt), to_dev(b, dt)
            ctx.sweep(ut, bt, nsweeps)
            assert ctx.last_error() == 0
            return float(np.sqrt(((to_np(ut).astype(LD) - ref) ** 2).sum() / (ref ** 2).sum()))

    digits = distance()
    monkeypatch.setenv("BRSMOOTH_MODE_SLICES", "0")
    assert digits <= distance()
