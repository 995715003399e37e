"""Alignment checks of the adjoint sweep: arrays that are not whole elements, and u_k or b off the
16-byte boundaries of a grid whose rows lie on them, are refused before anything is launched; a grid
of other rows takes element-aligned arrays and gives what it gives for aligned ones."""
import pytest

from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

NAMES = ("lam", "u_k", "b", "grad_b")


def call(lib, ctx, n, dt, shift_of=None, shift=0):
    """Status and updated arrays of one call, array `shift_of` moved by `shift` bytes."""
    import torch

    size = 8 if dt == "f64" else 4
    td = torch.float64 if dt == "f64" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(3)
    raw, ptr = {}, {}
    for name in NAMES:
        values = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64).to(td)
        raw[name] = torch.zeros(n * size + 64, dtype=torch.uint8, device="cuda")
        at = shift if name == shift_of else 0
        raw[name][at:at + n * size] = values.view(torch.uint8)
        ptr[name] = raw[name].data_ptr() + at
    ga = torch.zeros(3, dtype=torch.float64, device="cuda")
    rc = lib.brsmooth_adjoint_sweep(ctx.h, *(ptr[k] for k in NAMES), ga.data_ptr(), 0)
    torch.cuda.synchronize()
    out = [raw[k][(shift if k == shift_of else 0):][:n * size].clone() for k in ("lam", "grad_b")]
    return rc, out + [ga]


@pytest.mark.parametrize("dt", ["f64", "f32"])
def test_refused(brs, dt):  # noqa: F811
    size = 8 if dt == "f64" else 4
    with brs.Context(32, 6, 5, (1.0, 0.5, 0.25), block="line", method="jacobi", dtype=dt) as ctx:
        assert call(brs, ctx, 960, dt)[0] == brs.BRS_OK
        for name in NAMES:
            assert call(brs, ctx, 960, dt, name, size // 2)[0] == brs.BRS_ERR_ARG
        for name in ("u_k", "b"):
            assert call(brs, ctx, 960, dt, name, size)[0] == brs.BRS_ERR_ARG
        assert call(brs, ctx, 960, dt)[0] == brs.BRS_OK


@pytest.mark.parametrize("dt", ["f64", "f32"])
def test_ragged_rows_take_element_alignment(brs, dt):  # noqa: F811
    import torch

    size = 8 if dt == "f64" else 4
    with brs.Context(33, 6, 5, (1.0, 0.5, 0.25), block="line", method="jacobi", dtype=dt) as ctx:
        rc, ref = call(brs, ctx, 990, dt)
        assert rc == brs.BRS_OK
        for name in NAMES:
            assert call(brs, ctx, 990, dt, name, size // 2)[0] == brs.BRS_ERR_ARG
            rc, got = call(brs, ctx, 990, dt, name, size)
            assert rc == brs.BRS_OK
            assert all(torch.equal(x, y) for x, y in zip(got, ref))
