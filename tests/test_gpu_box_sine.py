"""Box sweeps in the box's sine basis (one fused pass) against the oracle's dense inverse, at
every side from 1 to 16 on every axis, odd box counts, and one context either side of the
longest side the form takes."""
import pytest

from gpu_common import TOL, rel_max_err
from test_gpu_box import brs, gpu_sweeps, inputs  # noqa: F401

pytestmark = pytest.mark.gpu

BOXES = [(1, 2, 3), (2, 3, 1), (3, 1, 2), (4, 5, 6), (5, 6, 4), (6, 4, 5), (7, 9, 8), (9, 8, 7),
         (8, 7, 9), (10, 3, 11), (11, 10, 3), (3, 11, 10), (12, 2, 13), (13, 12, 2), (2, 13, 12),
         (14, 2, 15), (15, 14, 2), (2, 15, 14), (16, 16, 2), (16, 2, 16), (2, 16, 16), (1, 1, 16),
         (16, 1, 1), (1, 16, 1), (8, 8, 2), (17, 2, 2), (2, 2, 17)]


@pytest.mark.parametrize("dt", ["f64", "f32"])
@pytest.mark.parametrize("method,omega", [("jacobi", 0.8), ("gs", 1.0), ("gs", 1.3)])
@pytest.mark.parametrize("box", BOXES, ids=lambda s: "x".join(map(str, s)))
def test_sides(brs, orc, box, method, omega, dt):  # noqa: F811
    counts = (7, 3, 5) if box[0] * box[1] * box[2] < 64 else (3, 3, 2)
    shape = tuple(n * c for n, c in zip(box, counts))
    a = (1.0, 0.1, 0.01)
    u, b = inputs(shape, dt)
    got = gpu_sweeps(brs, u, b, a, box, dt=dt, method=method, omega=omega, math="simt")[0]
    ref = orc.sweep(u, b, a, block="box", box=box, omega=omega,
                    method="jacobi" if method == "jacobi" else "gs_zebra")
    assert rel_max_err(got, ref) <= TOL[dt]
