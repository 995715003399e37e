"""Launch shapes of batched contexts of one patch set in one process: the tuner keeps them apart by
the kernel that runs them and by what the environment fixes, so no context gets a shape that its
kernel cannot run or that was never timed for it."""
import itertools

import numpy as np
import pytest

from gpu_common import to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

# (warps per CTA, CTAs per SM)
RING = {(4, 2), (4, 5), (8, 2)}
DIRECT = {(w, c) for w, c in itertools.product((4, 8, 16), (2, 4, 8)) if w * c <= 64}


def patches(n, seed):
    rng = np.random.default_rng(seed)
    return (4 * rng.integers(2, 17, (n, 3))).astype(np.int64)


def sweep(lib, dims):
    """Shape of a context of `dims` and the iterate of three Jacobi sweeps."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = int(dims.prod(axis=1).sum())
    rng = np.random.default_rng(7)
    u, b = to_dev(rng.uniform(-1, 1, n), "f32"), to_dev(rng.uniform(-1, 1, n), "f32")
    with lib.BatchedContext(dims, (1.0, 0.5, 0.25), method="jacobi", dtype="f32") as ctx:
        cfg = ctx.config()
        ctx.sweep(u, b, 3)
        assert ctx.last_error() == 0
        return cfg["kchunk"], (cfg["warps_per_cta"], cfg["ctas"] // sms), to_np(u)


@pytest.mark.parametrize("npatch", [3, 40, 300])
@pytest.mark.parametrize("first", ["direct", "ring"])
def test_each_kernel_has_its_own_shape(brs, npatch, first, monkeypatch):  # noqa: F811
    dims = patches(npatch, 100 * npatch + (first == "ring"))
    out = {}
    for form in (first, "ring" if first == "direct" else "direct"):
        monkeypatch.setenv("BRSMOOTH_BATCH_ASYNC", "1" if form == "ring" else "0")
        _, shape, out[form] = sweep(brs, dims)
        assert shape in (RING if form == "ring" else DIRECT)
    assert np.array_equal(out["direct"], out["ring"])


def test_fixed_chunks_are_kept(brs, monkeypatch):  # noqa: F811
    dims = patches(20, 5)
    ref = None
    for kc in (4, 16, 5, 32):
        monkeypatch.setenv("BRSMOOTH_BATCH_KC", str(kc))
        got, _, u = sweep(brs, dims)
        assert got == kc
        ref = u if ref is None else ref
        assert np.array_equal(u, ref)


def test_ring_depths_have_their_own_shapes(brs, monkeypatch):  # noqa: F811
    """The rings of all resident warps fit an SM: 20 warps do at 4 slots (8 KB each), not at 8."""
    dims = patches(300, 9)
    out = {}
    for stages in (4, 8):
        monkeypatch.setenv("BRSMOOTH_BATCH_STAGES", str(stages))
        _, (warps, ctas), out[stages] = sweep(brs, dims)
        assert warps * ctas * stages * 2048 <= 220 * 1024
    assert np.array_equal(out[4], out[8])
