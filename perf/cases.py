"""Timed workloads: block-relaxation sweeps through the package's public entry points.

Every workload is one call (or the few calls) that a program makes on data it already holds on
the GPU, with the contexts it keeps: single-grid sweeps (x-, y- and z-lines, xy-planes, boxes),
many-patch sweeps, levels with ghost exchange, FP32-in-FP64 defect correction, and the forward
and backward pass of the differentiable smoother.  Inputs are those of the convergence studies:
u0 and f uniform in [-1, 1], b = h^2 f.
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1208_1975_gb300 as brs

ISO = {"ax": 1.0, "ay": 1.0, "az": 1.0}


def _grid(name, block, method, dtype, n, sweeps, a=(1.0, 1.0, 1.0), **more):
    c = {"kind": "grid", "block": block, "method": method, "dtype": dtype, "nx": n[0], "ny": n[1],
         "nz": n[2], "sweeps": sweeps, "ax": a[0], "ay": a[1], "az": a[2]}
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    aniso = (1.0, 1.0, 0.01)
    return [
        # the smallest grid: a coarse level or a quick study, 10 sweeps from a zero guess
        _grid("line_f64_jacobi_32", "line", "jacobi", "f64", (32, 32, 32), 10, u0_zero=True),
        # one smoothing step (three sweeps) of one uneven patch, sides from the 64..96 patches
        _grid("line_f64_gs_patch", "line", "gs", "f64", (96, 88, 72), 3),
        # the headline sweep: one large grid in double precision, many sweeps per call
        _grid("line_f64_jacobi_256", "line", "jacobi", "f64", (256, 256, 256), 50),
        # the same grid in single precision, weak z coupling
        _grid("line_f32_jacobi_256", "line", "jacobi", "f32", (256, 256, 256), 50, aniso),
        # plane smoothing in single precision, many sweeps per call
        _grid("plane_f32_gs_256", "plane", "gs", "f32", (256, 256, 256), 50, aniso),
        # one sweep per call on a ragged grid: a smoother inside somebody else's cycle
        _grid("plane_f32_jacobi_1sweep", "plane", "jacobi", "f32", (200, 190, 180), 1, aniso),
        # plane smoothing in double precision, many sweeps per call
        _grid("plane_f64_jacobi_256", "plane", "jacobi", "f64", (256, 256, 256), 50, aniso),
        # spatial blocks in the paper's own size and precision, one smoothing step of a patch
        _grid("box8_f64_gs_96", "box", "gs", "f64", (96, 96, 96), 3, bx=8, by=8, bz=8),
        # spatial blocks on a large grid in single precision
        _grid("box8_f32_jacobi_256", "box", "jacobi", "f32", (256, 256, 256), 10, bx=8, by=8, bz=8),
        # 600 uneven patches of one refinement level swept as one stream of work
        dict(ISO, name="batched_f32_jacobi_600", kind="batched", method="jacobi", dtype="f32",
             npatch=600, lo=16, hi=64, step=8, sweeps=20),
        # gradients through 8 sweeps (gradient-checked runs are double), every iterate kept
        dict(ISO, name="adjoint_f64_128", kind="adjoint", dtype="f64", nx=128, ny=128, nz=128,
             sweeps=8),
        # a solve: single-precision plane sweeps inside double-precision defect correction
        {"name": "defect_plane_256", "kind": "defect", "block": "plane", "method": "gs", "nx": 256,
         "ny": 256, "nz": 256, "ax": 1.0, "ay": 0.1, "az": 0.01, "inner": 32, "rtol": 1e-10},
    ]


# ------------------------------------------------------------------------------ drawn cases

_COEFFS = ((1.0, 1.0, 1.0), (1.0, 1.0, 0.01), (1.0, 0.1, 0.01), (0.5, 1.0, 2.0))
_MAX_CELLS = 256 ** 3


def _size(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _dims(rng, lo, hi, most=_MAX_CELLS, xmax=512):
    n = [_size(rng, lo, min(hi, xmax)), _size(rng, lo, hi), _size(rng, lo, hi)]
    if rng.random() < 0.4:  # rows that start on 16-byte boundaries, as padded grids have them
        n = [(v + 3) // 4 * 4 for v in n]
    while n[0] * n[1] * n[2] > most:
        i = n.index(max(n))
        n[i] = max(lo, n[i] * 3 // 4)
    return n


def draw(rng):
    a = rng.choice(_COEFFS)
    kind = rng.choice(("line", "line", "line", "plane", "plane", "yline", "zline", "box", "box",
                       "batched", "level", "adjoint", "defect"))
    method = rng.choice(("jacobi", "gs"))
    dtype = rng.choice(("f64", "f32"))
    sweeps = rng.choice((1, 2, 3, 5, 10, 20, 50))
    if kind in ("line", "yline", "zline"):
        # FP32 Gauss-Seidel lines update in no fixed order, so drawn ones are Jacobi
        if dtype == "f32":
            method = "jacobi"
        return _grid(None, kind, method, dtype, _dims(rng, 16, 384), sweeps, a)
    if kind == "plane":
        most = _MAX_CELLS if dtype == "f32" else _MAX_CELLS // 2
        return _grid(None, kind, method, dtype, _dims(rng, 16, 384, most), sweeps, a)
    if kind == "box":
        box = rng.choice(((2, 2, 2), (4, 2, 2), (4, 4, 2), (4, 4, 4), (8, 4, 4), (8, 8, 4),
                          (8, 8, 8), (6, 5, 4), (3, 3, 3), (16, 4, 2)))
        n = [v // b * b if v >= b else b for v, b in zip(_dims(rng, 16, 256, _MAX_CELLS // 4), box)]
        return _grid(None, kind, method, dtype, n, min(sweeps, 10), a, bx=box[0], by=box[1],
                     bz=box[2])
    if kind == "batched":
        lo = rng.choice((8, 16, 24))
        return {"kind": "batched", "method": "jacobi", "dtype": dtype, "npatch": _size(rng, 32, 600),
                "lo": lo, "hi": rng.choice((48, 64)), "step": rng.choice((1, 4, 8)),
                "sweeps": min(sweeps, 20), "ax": a[0], "ay": a[1], "az": a[2]}
    if kind == "level":
        m = rng.choice((16, 24, 32, 48, 64, 72))
        return {"kind": "level", "method": "jacobi", "dtype": dtype, "px": rng.randint(1, 4),
                "py": rng.randint(1, 4), "pz": rng.randint(1, 4), "nx": m,
                "ny": m + rng.choice((-5, 0, 0, 8)), "nz": m + rng.choice((-3, 0, 0, 8)),
                "sweeps": min(sweeps, 5), "ax": a[0], "ay": a[1], "az": a[2]}
    if kind == "adjoint":
        n = _dims(rng, 16, 160, 128 ** 3)
        return {"kind": "adjoint", "dtype": dtype, "nx": n[0], "ny": n[1], "nz": n[2],
                "sweeps": rng.choice((4, 8)), "ax": a[0], "ay": a[1], "az": a[2]}
    n = 4 * _size(rng, 8, 40)
    return {"kind": "defect", "block": rng.choice(("plane", "plane", "line")), "method": "jacobi",
            "nx": n, "ny": n, "nz": n, "ax": 1.0, "ay": 0.1, "az": 0.01,
            "inner": rng.choice((8, 32)), "rtol": 1e-8}


# ------------------------------------------------------------------------------ inputs

def _uniform(gen, n, dtype=torch.float64):
    return torch.rand(n, generator=gen, device="cuda", dtype=dtype).mul_(2).sub_(1)


def _td(case):
    return torch.float64 if case.get("dtype", "f64") == "f64" else torch.float32


def _coef(case):
    return (case["ax"], case["ay"], case["az"])


def _patch_dims(case, seed):
    if case["kind"] == "level":
        P = (case["px"], case["py"], case["pz"])
        idx = lambda i, j, k: i + P[0] * (j + P[1] * k)  # noqa: E731
        nbr = []
        for k in range(P[2]):
            for j in range(P[1]):
                for i in range(P[0]):
                    nbr.append([idx(i - 1, j, k) if i else -1, idx(i + 1, j, k) if i + 1 < P[0] else -1,
                                idx(i, j - 1, k) if j else -1, idx(i, j + 1, k) if j + 1 < P[1] else -1,
                                idx(i, j, k - 1) if k else -1, idx(i, j, k + 1) if k + 1 < P[2] else -1])
        dims = np.array([[case["nx"], case["ny"], case["nz"]]] * len(nbr), dtype=np.int64)
        return dims, np.array(nbr, dtype=np.int64)
    # the set of patches belongs to the case: other seeds give other fields on the same patches
    r = random.Random("%d %d %d %d" % (case["npatch"], case["lo"], case["hi"], case["step"]))
    dims = [[r.randrange(case["lo"], case["hi"] + 1, case["step"]) for _ in range(3)]
            for _ in range(case["npatch"])]
    return np.array(dims, dtype=np.int64), None


def _fields(case, seed):
    """u0 and b (and the adjoint's target) as the program holds them, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] in ("batched", "level"):
        dims, _ = _patch_dims(case, seed)
        n, h = int(dims.prod(axis=1).sum()), 1.0 / (int(dims.max()) + 1)
        shape = (n,)
    else:
        shape = (case["nz"], case["ny"], case["nx"])
        h = 1.0 / (case["nx"] + 1)
    dt = _td(case)
    b = _uniform(gen, shape).mul_(h * h).to(dt)
    u = torch.zeros(shape, dtype=dt, device="cuda") if case.get("u0_zero") or case["kind"] == "defect" \
        else _uniform(gen, shape).to(dt)
    target = _uniform(gen, shape).to(dt) if case["kind"] == "adjoint" else None
    return u, b, target


def prepare(case, seed):
    u, b, target = _fields(case, seed)
    s = {"case": case, "u": u, "b": b}
    kind, a = case["kind"], _coef(case)
    if kind == "grid":
        s["ctx"] = brs.Context(case["nx"], case["ny"], case["nz"], a, block=case["block"],
                               method=case["method"], dtype=case["dtype"],
                               box=(case.get("bx", 0), case.get("by", 0), case.get("bz", 0)))
    elif kind in ("batched", "level"):
        dims, nbr = _patch_dims(case, seed)
        s["ctx"] = brs.BatchedContext(dims, a, method=case["method"], dtype=case["dtype"], nbr=nbr)
    elif kind == "defect":
        n = (case["nx"], case["ny"], case["nz"])
        s["outer"] = brs.Context(*n, a, block="line", method="jacobi", dtype="f64")
        s["inner"] = brs.Context(*n, a, block=case["block"], method=case["method"], dtype="f32")
    else:
        # a training loop's buffers: the trajectory u_0 .. u_K, the adjoint and the gradients
        s["ctx"] = brs.Context(case["nx"], case["ny"], case["nz"], a, block="line",
                               method="jacobi", dtype=case["dtype"])
        s["target"] = target
        s["traj"] = [u] + [torch.empty_like(u) for _ in range(case["sweeps"])]
        s["lam"], s["grad_b"] = torch.empty_like(u), torch.empty_like(u)
        s["grad_a"] = torch.empty(3, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("grid", "batched", "level"):
        # sweeps in place, as a smoother is called; the next pass smooths on
        s["ctx"].sweep(s["u"], s["b"], case["sweeps"])
        return s["u"]
    if kind == "defect":
        s["u"].zero_()  # each solve starts from the zero guess
        brs.defect_correction(s["outer"], s["inner"], s["u"], s["b"], rtol=case["rtol"],
                              inner_sweeps=case["inner"], max_outer=400)
        return s["u"]
    ctx, b, traj, lam, gb, ga = (s[k] for k in ("ctx", "b", "traj", "lam", "grad_b", "grad_a"))
    for k in range(case["sweeps"]):
        ctx.sweep(traj[k + 1].copy_(traj[k]), b, 1)
    torch.sub(traj[-1], s["target"], out=lam)  # gradient of 0.5 ||u_K - target||^2
    gb.zero_()
    ga.zero_()
    stream = torch.cuda.current_stream().cuda_stream
    for k in reversed(range(case["sweeps"])):
        rc = brs.brsmooth_adjoint_sweep(ctx.h, *(ctypes.c_void_p(t.data_ptr())
                                                 for t in (lam, traj[k], b, gb, ga)), stream)
        if rc != brs.BRS_OK:
            raise RuntimeError(brs.brsmooth_strerror(rc))
    return {"u": traj[-1], "grad_b": gb, "grad_u0": lam, "grad_a": ga}


# ------------------------------------------------------------------------------ work

def work(case):
    """Each input read once and each output written once; the multiplies and adds of the sweeps
    (gather, exact block solve by the cheapest factorised form, damped update)."""
    kind, size = case["kind"], 8 if case.get("dtype", "f64") == "f64" else 4
    if kind in ("batched", "level"):
        cells = int(_patch_dims(case, 0)[0].prod(axis=1).sum())
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    line = 12.0  # 4 neighbours (2 adds, 2 FMAs), two elimination FMAs, damped update FMA
    if kind == "grid":
        per = line
        if case["block"] == "plane":  # two fast sine transforms along x besides
            per = line + 2 * 5 * math.log2(2 * case["nx"])
        if case["block"] == "box":  # the block's sine basis, by axis, there and back
            per = 12.0 + 2.0 * (case["bx"] + case["by"] + case["bz"])
        return {"bytes": 3.0 * cells * size, "flops": per * cells * case["sweeps"]}
    if kind in ("batched", "level"):
        return {"bytes": 3.0 * cells * size, "flops": line * cells * case["sweeps"]}
    if kind == "defect":
        # b read, u written, and at least one correction: a residual, its sweeps, an update
        return {"bytes": 2.0 * cells * 8, "flops": cells * (14.0 + line * case["inner"])}
    # u0, b, the loss gradient in; u, grad_b, grad_u0 out; forward sweep and reverse step
    return {"bytes": 6.0 * cells * size, "flops": cells * case["sweeps"] * (line + 3 * line)}


# ------------------------------------------------------------------------------ 64-bit values

def _sine(n):
    i = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    return math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi * torch.outer(i, i) / (n + 1))


def _eig(n):
    i = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    return 4.0 * torch.sin(math.pi * i / (2 * (n + 1))) ** 2


def _on(M, x, axis):
    """M applied along one axis (0 = z, 1 = y, 2 = x of the last three) of x."""
    return torch.movedim(torch.movedim(x, axis - 3, -1) @ M.T, -1, axis - 3)


def _apply(u, a):
    """A u on (..., nz, ny, nx), zero outside."""
    ax, ay, az = a
    r = (2.0 * (ax + ay + az)) * u
    r[..., :, 1:] -= ax * u[..., :, :-1]
    r[..., :, :-1] -= ax * u[..., :, 1:]
    r[..., :, 1:, :] -= ay * u[..., :, :-1, :]
    r[..., :, :-1, :] -= ay * u[..., :, 1:, :]
    r[..., 1:, :, :] -= az * u[..., :-1, :, :]
    r[..., :-1, :, :] -= az * u[..., 1:, :, :]
    return r


def _line_inverse(n, a, axis=0):
    """Inverse of the line block along x (axis 0), y or z."""
    off = a[axis]
    M = torch.diag(torch.full((n,), 2.0 * sum(a), dtype=torch.float64, device="cuda"))
    e = torch.full((n - 1,), -off, dtype=torch.float64, device="cuda")
    return torch.linalg.inv(M + torch.diag(e, 1) + torch.diag(e, -1))


def _box_solver(b, a, n):
    """r -> M^{-1} r for boxes b = (bx, by, bz) of a grid n = (nx, ny, nz)."""
    S = [_sine(v) for v in b]
    lam = (a[0] * _eig(b[0])[None, None, :] + a[1] * _eig(b[1])[None, :, None]
           + a[2] * _eig(b[2])[:, None, None])

    def solve(r):
        t = r.reshape(n[2] // b[2], b[2], n[1] // b[1], b[1], n[0] // b[0], b[0])
        t = t.permute(0, 2, 4, 1, 3, 5)
        for ax in range(3):
            t = _on(S[ax], t, 2 - ax)
        t = t / lam
        for ax in range(3):
            t = _on(S[ax], t, 2 - ax)
        return t.permute(0, 3, 1, 4, 2, 5).reshape(r.shape)
    return solve


def _solver(case):
    a, n, block = _coef(case), (case["nx"], case["ny"], case["nz"]), case["block"]
    if block in ("line", "yline", "zline"):
        d = ("line", "yline", "zline").index(block)
        inv = _line_inverse(n[d], a, d)
        return lambda r: _on(inv, r, 2 - d)
    if block == "plane":
        Sx, Sy = _sine(n[0]), _sine(n[1])
        lam = a[0] * _eig(n[0])[None, :] + a[1] * _eig(n[1])[:, None] + 2.0 * a[2]
        return lambda r: _on(Sx, _on(Sy, _on(Sy, _on(Sx, r, 2), 1) / lam, 1), 2)
    return _box_solver((case["bx"], case["by"], case["bz"]), a, n)


def _colours(case):
    """The two sets of cells that a two-colour sweep updates in turn."""
    ijk = [torch.arange(case[k], device="cuda") for k in ("nx", "ny", "nz")]
    block = case["block"]
    if block == "box":
        ijk = [v // case[k] for v, k in zip(ijk, ("bx", "by", "bz"))]
    i, j, k = ijk[0][None, None, :], ijk[1][None, :, None], ijk[2][:, None, None]
    c = {"line": 0 * i + j + k, "yline": i + 0 * j + k, "zline": i + j + 0 * k,
         "plane": 0 * i + 0 * j + k, "box": i + j + k}[block] % 2
    return c == 0, c == 1


def _exact_grid(case, u, b):
    a, solve = _coef(case), _solver(case)
    if case["method"] == "jacobi":
        for _ in range(case["sweeps"]):
            u = u + 0.8 * solve(b - _apply(u, a))
        return u
    for _ in range(case["sweeps"]):
        for mask in _colours(case):
            u = torch.where(mask, u + solve(b - _apply(u, a)), u)
    return u


def _exact_patches(case, u, b, seed):
    a = _coef(case)
    if case["kind"] == "level":
        P, n = (case["px"], case["py"], case["pz"]), (case["nx"], case["ny"], case["nz"])

        def whole(x):  # patches -> the grid they tile
            return x.reshape(P[2], P[1], P[0], n[2], n[1], n[0]).permute(0, 3, 1, 4, 2, 5).reshape(
                P[2] * n[2], P[1] * n[1], P[0] * n[0])
        inv, g, r = _line_inverse(n[0], a), whole(u), whole(b)
        for _ in range(case["sweeps"]):
            d = (r - _apply(g, a)).reshape(-1, n[0]) @ inv
            g = g + 0.8 * d.reshape(g.shape)
        return g.reshape(P[2], n[2], P[1], n[1], P[0], n[0]).permute(0, 2, 4, 1, 3, 5).reshape(-1)
    dims, _ = _patch_dims(case, seed)
    out, at, inv = torch.empty_like(u), 0, {}
    for nx, ny, nz in dims.tolist():
        n = nx * ny * nz
        if nx not in inv:
            inv[nx] = _line_inverse(nx, a)
        p, r = u[at:at + n].reshape(nz, ny, nx), b[at:at + n].reshape(nz, ny, nx)
        for _ in range(case["sweeps"]):
            p = p + 0.8 * ((r - _apply(p, a)) @ inv[nx])
        out[at:at + n] = p.reshape(-1)
        at += n
    return out


def _exact_adjoint(case, u, b, target):
    a = torch.tensor(_coef(case), dtype=torch.float64, device="cuda", requires_grad=True)
    u0, b = u.requires_grad_(True), b.requires_grad_(True)
    n = case["nx"]
    off = torch.diag(torch.ones(n - 1, dtype=torch.float64, device="cuda"), 1)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    inv = torch.linalg.inv(2.0 * a.sum() * eye - a[0] * (off + off.T))
    pad = torch.nn.functional.pad
    v = u0
    for _ in range(case["sweeps"]):
        w = pad(v[None], (1, 1, 1, 1, 1, 1))[0]
        near = (a[0] * (w[1:-1, 1:-1, :-2] + w[1:-1, 1:-1, 2:]) + a[1] * (w[1:-1, :-2, 1:-1] + w[1:-1, 2:, 1:-1])
                + a[2] * (w[:-2, 1:-1, 1:-1] + w[2:, 1:-1, 1:-1]))
        v = v + 0.8 * ((b - 2.0 * a.sum() * v + near) @ inv)
    gb, gu, ga = torch.autograd.grad(v, (b, u0, a), v.detach() - target)
    return {"u": v.detach(), "grad_b": gb, "grad_u0": gu, "grad_a": ga}


def exact(case, seed):
    u, b, target = _fields(case, seed)
    u, b = u.double(), b.double()
    kind, a = case["kind"], _coef(case)
    if kind == "grid":
        return _exact_grid(case, u, b)
    if kind in ("batched", "level"):
        return _exact_patches(case, u, b, seed)
    if kind == "adjoint":
        return _exact_adjoint(case, u, b, target.double())
    S = [_sine(case[k]) for k in ("nx", "ny", "nz")]
    for d in range(3):
        b = _on(S[d], b, 2 - d)
    b = b / (a[0] * _eig(case["nx"])[None, None, :] + a[1] * _eig(case["ny"])[None, :, None]
             + a[2] * _eig(case["nz"])[:, None, None])
    for d in range(3):
        b = _on(S[d], b, 2 - d)
    return b
