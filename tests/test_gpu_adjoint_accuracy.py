"""FP64 gradients through 8 x-line Jacobi sweeps against extended precision, beside the same reverse
sweep in FP64 as it is defined (mu = M^{-1} lambda by Thomas, lambda - omega A mu, fused multiply-adds)."""
import numpy as np
import pytest

from gpu_common import to_dev, to_np
from test_gpu_box import brs  # noqa: F401

pytestmark = pytest.mark.gpu

LD = np.longdouble
SWEEPS, OMEGA = 8, 0.8


def beside(v, axis):
    """Sum of the two neighbours along an axis, zero outside."""
    w = np.moveaxis(v, axis, 0)
    s = np.zeros_like(w)
    s[1:] += w[:-1]
    s[:-1] += w[1:]
    return np.moveaxis(s, 0, axis)


def gradients(u0, b, target, a, ft):
    """grad_u0 and grad_b of 0.5 ||u_K - target||^2, every operation rounded to ft."""
    def fma(x, y, z):
        return (np.asarray(x, LD) * np.asarray(y, LD) + np.asarray(z, LD)).astype(ft)

    ax, ay, az = (ft(v) for v in a)
    d, om = ft(2) * (ax + ay + az), ft(OMEGA)
    nx = u0.shape[2]
    p = np.empty(nx, ft)
    p[0] = ft(1) / d
    for i in range(1, nx):
        p[i] = ft(1) / (d - ax * ax * p[i - 1])

    def solve(r):
        w = r.astype(ft).copy()
        for i in range(1, nx):
            w[..., i] = fma(ax * p[i - 1], w[..., i - 1], w[..., i])
        for i in range(nx - 2, -1, -1):
            w[..., i] = fma(ax * p[i + 1], w[..., i + 1], w[..., i])
        return p * w

    u, b = u0.astype(ft), b.astype(ft)
    for _ in range(SWEEPS):
        x = solve(fma(az, beside(u, 0), fma(ay, beside(u, 1), b)))
        u = fma(om, x, (ft(1) - om) * u)
    lam, gb = u - target.astype(ft), np.zeros_like(u)
    for _ in range(SWEEPS):
        mu = solve(lam)
        A = fma(-az, beside(mu, 0), fma(-ay, beside(mu, 1), fma(-ax, beside(mu, 2), d * mu)))
        lam, gb = fma(-om, A, lam), fma(om, mu, gb)
    return lam, gb


@pytest.mark.parametrize("a", [(1.0, 1.0, 1.0), (0.5, 1.0, 2.0)], ids=str)
@pytest.mark.parametrize("n", [(40, 30, 20), (33, 24, 25)], ids=lambda s: "x".join(map(str, s)))
def test_no_further_than_the_definition(brs, n, a):  # noqa: F811
    """The two round in other places (elimination from both ends, omega and the pivots folded into the
    right-hand sides): emulated on the CPU, at these sizes and coefficients and three seeds, the kernels'
    operations come to 1.07 .. 1.33 times the definition's 2-norm error.  A tenth more is allowed for
    other fields."""
    import torch

    rng = np.random.default_rng(5)
    u0, b, target = (rng.uniform(-1, 1, n[::-1]) for _ in range(3))
    b /= (n[0] + 1) ** 2
    bt, ut = to_dev(b, "f64").requires_grad_(True), to_dev(u0, "f64").requires_grad_(True)
    d = brs.block_smooth(bt, ut, torch.tensor(a, dtype=torch.float64, device="cuda"), SWEEPS,
                         ckpt=SWEEPS) - to_dev(target, "f64")
    (0.5 * (d * d).sum()).backward()
    exact = gradients(u0, b, target, a, LD)
    plain = gradients(u0, b, target, a, np.float64)
    for got, ref, ex in zip((to_np(ut.grad), to_np(bt.grad)), plain, exact):
        def distance(v):
            return float(np.sqrt(((v.astype(LD) - ex) ** 2).sum()))
        assert distance(got) <= 1.45 * distance(ref)
