"""One context swept on more buffers than it keeps tensor maps for: every call sees its own u and
b, whatever the cache of maps has dropped or moved."""
import pytest

from brs_inputs import initial_guess, rhs
from gpu_common import to_dev
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["jacobi", "gs"])
def test_more_buffers_than_cached_maps(brs, method):  # noqa: F811
    import torch

    n = 32
    us = [to_dev(initial_guess((n, n, n), seed=100 + q), "f32") for q in range(40)]
    bs = [to_dev(rhs((n, n, n), seed=200 + q), "f32") for q in range(40)]
    with brs.Context(n, n, n, (1.0, 1.0, 1.0), block="line", method=method, dtype="f32") as ctx:
        for _ in range(2):
            for u, b in zip(us, bs):
                ctx.sweep(u, b, 1)
        torch.cuda.synchronize()
        assert ctx.last_error() == 0
    if method == "gs":
        return  # chaotic order: no second run to compare with
    for q, (u, b) in enumerate(zip(us, bs)):
        ref = to_dev(initial_guess((n, n, n), seed=100 + q), "f32")
        with brs.Context(n, n, n, (1.0, 1.0, 1.0), block="line", method=method, dtype="f32") as ctx:
            ctx.sweep(ref, b, 1)
            ctx.sweep(ref, b, 1)
            assert torch.equal(u, ref)
