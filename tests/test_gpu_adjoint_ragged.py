"""FP64 adjoint sweeps at rows that end inside a chunk of 32 cells, planes that do not fill the
z-chunks, and lines of one cell, against the oracle's reverse-mode gradients; twice on one context,
whose reduction leaves its counter ready for the next call."""
import numpy as np
import pytest

from gpu_common import rel_max_err, to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(33, 17, 37), (97, 30, 65), (1, 5, 9), (32, 1, 70), (64, 9, 1), (300, 5, 11)]
SWEEPS, A = 4, (1.0, 0.7, 0.3)


@pytest.mark.parametrize("omega", [0.8, 1.3])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_matches_oracle(brs, orc, shape, omega):  # noqa: F811
    import torch

    nx, ny, nz = shape
    rng = np.random.default_rng(5)
    u0, b, target = (rng.uniform(-1, 1, (nz, ny, nx)) for _ in range(3))
    _, gu, gb, ga = orc.adjoint_gradients(u0, b, A, SWEEPS, target, block="line", omega=omega)
    bt = to_dev(b, "f64")
    with brs.Context(nx, ny, nz, A, block="line", method="jacobi", dtype="f64", omega=omega) as ctx:
        traj = [to_dev(u0, "f64")]
        for _ in range(SWEEPS):
            traj.append(traj[-1].clone())
            ctx.sweep(traj[-1], bt, 1)
        for _ in range(2):
            lam = traj[-1] - to_dev(target, "f64")
            grad_b, grad_a = torch.zeros_like(lam), torch.zeros(3, dtype=torch.float64, device="cuda")
            for k in reversed(range(SWEEPS)):
                rc = brs.brsmooth_adjoint_sweep(ctx.h, lam.data_ptr(), traj[k].data_ptr(), bt.data_ptr(),
                                                grad_b.data_ptr(), grad_a.data_ptr(), 0)
                assert rc == brs.BRS_OK
            assert rel_max_err(to_np(lam), gu) <= 1e-11
            assert rel_max_err(to_np(grad_b), gb) <= 1e-11
            scale = float(np.abs(ga).max())
            assert np.abs(grad_a.cpu().numpy() - ga).max() <= 1e-11 * scale
