"""The calls a user of this package makes, with the sizes they make them at.

Each case is one pass through the public entry points on inputs shaped like the
scans of ``synthetic.py``: the FFP operators A and A^T (2-D and 3-D), their
gradients, the Core Stage, and the two reconstructions built on them.

``exact`` restates each result from the model's formulas in 64-bit torch, with
none of the package's own arithmetic.
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_2505_22797_gb300 import api, autograd
from paper_2505_22797_gb300 import synthetic as syn

DEV = "cuda"
F64 = torch.float64
DTYPES = {"f32": torch.float32, "f64": torch.float64}
TILTED = [[2.4e-3, 3e-4], [3e-4, 2.6e-3]]  # selection field turned against the grid's axes


def listed():
    return [
        # One short period of the scanner's Lissajous scan on a preview grid: the smallest call,
        # made once per frame of a live view.
        dict(name="forward_32", kind="forward", nx=32, ny=32, T=1632, traj="lissajous", fov=24.0,
             dtype="f32", n_ch=2, tilt=False),
        # The benchmark's operator pair: 128 x 128 spiral scan, as a solver's inner loop or a
        # simulation applies them.
        dict(name="forward_128", kind="forward", nx=128, ny=128, T=65536, traj="spiral", fov=24.0,
             dtype="f32", n_ch=2, tilt=False),
        dict(name="adjoint_128", kind="adjoint", nx=128, ny=128, T=65536, traj="spiral", fov=24.0,
             dtype="f32", n_ch=2, tilt=False),
        # One receive channel, a selection field that is not aligned with the grid, and sizes that
        # fit no tile.
        dict(name="adjoint_tilted", kind="adjoint", nx=97, ny=113, T=20011, traj="lissajous", fov=24.0,
             dtype="f32", n_ch=1, tilt=True),
        # The largest configured scan: backprojection of 2^20 samples onto 512 x 512 voxels.
        dict(name="adjoint_512", kind="adjoint", nx=512, ny=512, T=1 << 20, traj="excited", fov=48.0,
             dtype="f32", n_ch=2, tilt=False),
        # Calibration of the particle parameter together with the image: forward and backward
        # through torch.autograd.
        dict(name="gradient_256", kind="gradient", nx=256, ny=256, T=262144, traj="lissajous", fov=24.0,
             dtype="f32", n_ch=2, tilt=False),
        # The plain FP64 method: A, then A^T of its result (one normal product).
        dict(name="normal_f64_64", kind="normal", nx=64, ny=48, T=3000, traj="spiral", fov=24.0,
             dtype="f64", n_ch=2, tilt=False),
        # A whole reconstruction with A as the data-fidelity operator.
        dict(name="recon_128", kind="recon", nx=128, ny=128, T=65536, traj="spiral", fov=24.0,
             dtype="f32", n_ch=2, tilt=False, n_iter=4, n_cg=5),
        # The paper's two-stage reconstruction on its 100 x 100 grid: Core Stage to the paper's
        # tolerance, then the deconvolution of its trace.
        dict(name="two_stage_100", kind="two_stage", nx=100, ny=100, T=1632, traj="lissajous", fov=24.0,
             dtype="f32", n_iter=10, n_cg=5),
        # The Core Stage of the largest scan (binning, right-hand side and CG steps).
        dict(name="core_512", kind="core", nx=512, ny=512, T=1 << 20, traj="excited", fov=48.0,
             dtype="f32", gamma=1e-7, steps=20, scaled=False),
        # The Core Stage in three dimensions.
        dict(name="core3_48", kind="core3", nx=48, ny=48, nz=24, T=65536, dtype="f32", gamma=1e-7, steps=20,
             scaled=False),
        # The 3-D operators: A, and A^T of the measured signal.
        dict(name="pair3_48", kind="pair3", nx=48, ny=48, nz=24, T=65536, dtype="f32", n_ch=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _aspect(rng, n, lo, hi):
    return max(lo, min(hi, int(round(n * rng.uniform(0.75, 1.33)))))


def draw(rng):
    kind = rng.choice(["forward", "adjoint", "forward", "adjoint", "gradient", "normal", "recon",
                       "two_stage", "core", "core3", "pair3"])
    traj = rng.choice(["lissajous", "spiral", "excited"])
    if kind in ("forward", "adjoint"):
        nx = _log(rng, 24, 512)
        ny = _aspect(rng, nx, 20, 512)
        T = _log(rng, 1000, 1 << 20)
        return dict(kind=kind, nx=nx, ny=ny, T=T, traj=traj, fov=rng.choice([24.0, 24.0, 48.0]), dtype="f32",
                    n_ch=rng.choice([1, 2, 2]), tilt=rng.random() < 0.25)
    if kind == "gradient":
        nx = _log(rng, 48, 256)
        return dict(kind=kind, nx=nx, ny=_aspect(rng, nx, 40, 256), T=_log(rng, 4096, 262144), traj=traj,
                    fov=24.0, dtype="f32", n_ch=2, tilt=rng.random() < 0.25)
    if kind == "normal":
        nx = rng.randint(24, 72)
        return dict(kind=kind, nx=nx, ny=_aspect(rng, nx, 24, 72), T=_log(rng, 1000, 6000), traj=traj, fov=24.0,
                    dtype="f64", n_ch=rng.choice([1, 2, 2]), tilt=rng.random() < 0.25)
    if kind == "recon":
        nx = _log(rng, 32, 128)
        return dict(kind=kind, nx=nx, ny=_aspect(rng, nx, 32, 128), T=_log(rng, 1632, 65536), traj=traj, fov=24.0,
                    dtype="f32", n_ch=2, tilt=False, n_iter=rng.randint(2, 4), n_cg=rng.randint(3, 5))
    if kind == "two_stage":
        nx = _log(rng, 21, 100)
        return dict(kind=kind, nx=nx, ny=_aspect(rng, nx, 21, 100), T=_log(rng, 1632, 16384), traj=traj, fov=24.0,
                    dtype="f32", n_iter=rng.randint(4, 10), n_cg=rng.randint(3, 5))
    if kind == "core":
        nx = _log(rng, 32, 512)
        return dict(kind=kind, nx=nx, ny=_aspect(rng, nx, 32, 512), T=_log(rng, 4096, 1 << 20), traj=traj, fov=24.0,
                    dtype="f32", gamma=1e-7, steps=rng.randint(10, 20), scaled=False)
    nx = rng.randint(16, 48)
    ny, nz = rng.randint(16, 48), rng.randint(8, 24)
    T = _log(rng, 4096, 65536)
    if kind == "core3":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, T=T, dtype="f32", gamma=1e-7, steps=rng.randint(10, 20),
                    scaled=False)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, T=T, dtype="f32", n_ch=rng.choice([2, 3, 3]))


# ---------------------------------------------------------------------------
# Inputs

def _model(case):
    if "nz" in case:
        return syn.default_model3(n_ch=case.get("n_ch", 3))
    m = syn.default_model(n_ch=case.get("n_ch", 2))
    return dict(m, G=TILTED) if case.get("tilt") else m


def _grid(case):
    if "nz" in case:
        return syn.box_grid3(case["nx"], case["ny"], case["nz"])
    return syn.square_grid(case["nx"], case["fov"], case["ny"])


def _trajectory(case, rng):
    T = case["T"]
    if "nz" in case:
        r, v = syn.lissajous3(T, 17, 16, 15)
        start = int(rng.integers(0, T))  # where in the period the record begins
        return np.roll(r, -start, axis=0), np.roll(v, -start, axis=0)
    amp = case["fov"] / 2
    if case["traj"] == "lissajous":
        return syn.lissajous(T, 17, 16, amp=amp, phase=float(rng.uniform(0, 2 * math.pi)))
    if case["traj"] == "excited":
        r, v = syn.lissajous_excited(T, 17, 16, amp, 1.5, 25.0)
        start = int(rng.integers(0, T))
        return np.roll(r, -start, axis=0), np.roll(v, -start, axis=0)
    r, v = syn.spiral(T, min(32.0, max(4.0, T / 512)), radius=amp)
    th = float(rng.uniform(0, 2 * math.pi))
    rot = np.array([[math.cos(th), math.sin(th)], [-math.sin(th), math.cos(th)]])
    return r @ rot, v @ rot


def _phantom(case, grid, rng):
    if "nz" in case:
        c = syn.ellipsoids(grid, rng)
    else:
        c = syn.point_sources(syn.ellipses(grid, rng, semi=(case["fov"] / 16, case["fov"] / 4)), rng)
    if not c.any():
        c[tuple(n // 2 for n in c.shape)] = 1.0
    return c


def _measured(case, model, grid, r, v, rng):
    """The signal of a few dozen particle spots, with 1 % noise (64-bit torch)."""
    fov = [case["fov"], case["fov"]] if "nz" not in case else [24.0, 24.0, 12.0]
    n = 48
    spots = torch.as_tensor(rng.uniform(-0.35, 0.35, (n, len(fov))) * np.array(fov), device=DEV)
    amount = torch.as_tensor(rng.uniform(0.5, 2.0, n) * 100.0, device=DEV)
    s = _sweep(model, spots, r.double(), v.double(), c=amount)["s"]
    noise = torch.as_tensor(rng.standard_normal(tuple(s.shape), dtype=np.float32), device=DEV)
    return s + 0.01 * s.abs().max() * noise.double()


def prepare(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, case["nx"], case["T"]])
    dt = DTYPES[case["dtype"]]
    st = dict(case=dict(case), model=_model(case), grid=_grid(case))
    r, v = _trajectory(case, rng)
    st["r"] = torch.as_tensor(np.ascontiguousarray(r), device=DEV).to(dt)
    st["v"] = torch.as_tensor(np.ascontiguousarray(v), device=DEV).to(dt)
    kind, model, grid = case["kind"], st["model"], st["grid"]
    if kind in ("forward", "gradient", "normal", "pair3"):
        st["c"] = torch.as_tensor(_phantom(case, grid, rng), device=DEV).to(dt).contiguous()
    if kind not in ("forward", "normal"):
        st["s"] = _measured(case, model, grid, st["r"], st["v"], rng).to(dt).contiguous()
    if kind == "gradient":
        st["c"].requires_grad_(True)
        st["beta"] = torch.tensor(model["beta"], dtype=F64, device=DEV, requires_grad=True)
    if kind == "recon":
        st["nu0"] = _nu0_A(model, grid, st["r"], st["v"])
    if kind == "two_stage":
        k = _trace_kernel(model, grid)
        ny, nx = grid["ny"], grid["nx"]
        st["nu0"] = 1e-3 * float((k[ny // 2:ny // 2 + ny, nx // 2:nx // 2 + nx] ** 2).sum())
    return st


# ---------------------------------------------------------------------------
# One pass

def run(st):
    case, model, grid, r, v = st["case"], st["model"], st["grid"], st["r"], st["v"]
    kind = case["kind"]
    if kind == "forward":
        return api.mpi_forward(model, grid, r, v, st["c"])
    if kind == "adjoint":
        return api.mpi_adjoint(model, grid, r, v, st["s"])
    if kind == "normal":
        s = api.mpi_forward(model, grid, r, v, st["c"])
        return {"s": s, "c": api.mpi_adjoint(model, grid, r, v, s)}
    if kind == "gradient":
        s = autograd.mpi_forward_autograd(st["c"], st["beta"], model, grid, r, v)
        gc, gb = torch.autograd.grad(s, (st["c"], st["beta"]), grad_outputs=s.detach() - st["s"])
        return {"s": s.detach(), "dc": gc, "dbeta": gb}
    if kind == "recon":
        return api.mpi_pnp_solve(model, grid, r, v, st["s"], case["n_iter"], case["n_cg"], st["nu0"])
    if kind == "two_stage":
        A, u = api.mpi_grid(grid, r, v, st["s"], gamma=1e-7, max_iter=10000, rel_tol=1e-3, lap_scaled=True)
        rho = api.mpi_pnp_solve(model, grid, None, None, u, case["n_iter"], case["n_cg"], st["nu0"],
                                op=api.MPI_OP_CONV)
        return {"A": A, "rho": rho}
    if kind == "core":
        A, u = api.mpi_grid(grid, r, v, st["s"], gamma=case["gamma"], max_iter=case["steps"], rel_tol=0.0,
                            lap_scaled=case["scaled"])
        return {"A": A, "u": u}
    if kind == "core3":
        A, u = api.mpi_grid3(grid, r, v, st["s"], gamma=case["gamma"], max_iter=case["steps"], rel_tol=0.0,
                             lap_scaled=case["scaled"])
        return {"A": A, "u": u}
    if kind == "pair3":
        return {"s": api.mpi_forward3(model, grid, r, v, st["c"]),
                "c": api.mpi_adjoint3(model, grid, r, v, st["s"])}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# What a pass cannot do without

def _voxels(case):
    return case["nx"] * case["ny"] * case.get("nz", 1)


def _operator_flops(case):
    """One application of A or A^T: the direct sum over all pairs, or, where that is less, the
    same sums as convolutions with the kernel's three entries on a zero-padded grid of a quarter
    of its core radius with 10 x 10-point interpolation at the samples."""
    N, T = _voxels(case), case["T"]
    direct = (12 if "nz" not in case else 19) * N * T
    if "nz" in case or case["dtype"] != "f32":
        return direct
    side = case["fov"] * syn.BETA_1MM * syn.G_MM / 0.25
    m = (2 * side) ** 2
    return min(direct, 3 * 2.5 * m * math.log2(m) + 600 * T)


def work(case):
    N, T, kind = _voxels(case), case["T"], case["kind"]
    size = 4 if case["dtype"] == "f32" else 8
    dim = 3 if "nz" in case else 2
    n_ch = case.get("n_ch", dim)
    traj, sig = 2 * dim * T * size, n_ch * T * size
    op = _operator_flops(case)
    if kind in ("forward", "adjoint"):
        return {"bytes": traj + sig + N * size, "flops": op}
    if kind == "normal":
        return {"bytes": traj + sig + 2 * N * size, "flops": 2 * op}
    if kind == "gradient":
        return {"bytes": traj + 2 * sig + 2 * N * size, "flops": 3 * op}
    if kind == "pair3":
        return {"bytes": traj + 2 * sig + 2 * N * size, "flops": 2 * op}
    if kind == "recon":
        return {"bytes": traj + sig + N * size, "flops": 2 * op * (case["n_iter"] * (case["n_cg"] + 1) + 0.5)}
    comp = dim * dim
    # per CG step and unknown: two Laplacians, four vector updates and two inner products in
    # pairs of words; per sample the interpolation and its transpose on 2^dim nodes
    step = N * comp * 60 + T * comp * 2 ** dim * 4
    if kind in ("core", "core3"):
        return {"bytes": traj + sig + (comp + 1) * N * size, "flops": case["steps"] * step}
    conv = 2 * 2.5 * 4 * N * math.log2(4 * N)
    return {"bytes": traj + sig + (comp + 1) * N * size,
            "flops": 40 * step + case["n_iter"] * (case["n_cg"] + 1) * 2 * conv}


# ---------------------------------------------------------------------------
# The same results in 64 bits

def _coth_series(n):
    """c_1..c_n of coth z - 1/z = sum c_k z^(2k-1), from the Bernoulli numbers."""
    B = [Fraction(1)]
    for m in range(1, 2 * n + 1):
        B.append(-sum(Fraction(math.comb(m + 1, j)) * B[j] for j in range(m)) / (m + 1))
    return [float(Fraction(4) ** k * B[2 * k] / math.factorial(2 * k)) for k in range(1, n + 1)]


_C = _coth_series(16)


def _poly(u, coef):
    acc = torch.full_like(u, coef[-1])
    for a in reversed(coef[:-1]):
        acc = acc * u + a
    return acc


def _scalars(u, slope=False):
    """(a, d) with K(y) = a I + d y y^T and u = |y|^2, or with ``slope`` (L', L''/z)."""
    near = u < 0.25
    w = torch.where(near, torch.ones_like(u), u)
    z = w.sqrt()
    q = torch.exp(-2 * z)
    coth, csch2 = (1 + q) / (1 - q), 4 * q / (1 - q) ** 2
    lp = 1 / w - csch2
    if slope:
        e = (2 * coth * csch2 - 2 / (w * z)) / z
        return (torch.where(near, _poly(u, [(2 * k + 1) * c for k, c in enumerate(_C)]), lp),
                torch.where(near, _poly(u, [(2 * k + 2) * (2 * k + 3) * c for k, c in enumerate(_C[1:])]), e))
    a = coth / z - 1 / w
    return (torch.where(near, _poly(u, _C), a),
            torch.where(near, _poly(u, [(2 * k + 2) * c for k, c in enumerate(_C[1:])]), (lp - a) / w))


def _centres(grid):
    axes = [grid["%s0" % q] + (torch.arange(grid["n" + q], dtype=F64, device=DEV) + 0.5) * grid["d" + q]
            for q in "xyz" if "n" + q in grid]
    mesh = torch.meshgrid(*reversed(axes), indexing="ij")
    return torch.stack([m.reshape(-1) for m in reversed(mesh)], 1)


def _sweep(model, x, r, v, c=None, s=None, beta_of=None):
    """One pass over all (voxel, sample) pairs: s = A c, A^T s, and with ``beta_of`` (an image)
    d/dbeta <s, A(image)>."""
    B = float(model["beta"]) * torch.tensor(model["G"], dtype=F64, device=DEV)
    P = torch.tensor(model["p"], dtype=F64, device=DEV)
    X, R, W = x @ B.T, r @ B.T, v @ B.T
    N, T, dim = X.shape[0], R.shape[0], X.shape[1]
    out = {}
    if c is not None:
        out["s"] = torch.empty((P.shape[0], T), dtype=F64, device=DEV)
    if s is not None:
        out["c"] = torch.zeros(N, dtype=F64, device=DEV)
        U = s.T @ P
    slope = 0.0
    step = max(1, (1 << 25) // N)
    for t in range(0, T, step):
        e = slice(t, min(T, t + step))
        y = [X[None, :, i] - R[e, i, None] for i in range(dim)]
        u = sum(q * q for q in y)
        yW = sum(q * W[e, i, None] for i, q in enumerate(y))
        if c is not None or s is not None:
            a, d = _scalars(u)
            if c is not None:
                f = d * yW
                O = (a @ c)[:, None] * W[e] + torch.stack([(f * q) @ c for q in y], 1)
                out["s"][:, e] = (O @ P.T).T
            if s is not None:
                yU = sum(q * U[e, i, None] for i, q in enumerate(y))
                out["c"] += a.T @ (U[e] * W[e]).sum(1) + (d * yW * yU).sum(0)
                if beta_of is not None:
                    del a, d
                    lp, ez = _scalars(u, slope=True)
                    slope += float((((lp * (U[e] * W[e]).sum(1)[:, None] + ez * yW * yU)) @ beta_of).sum())
    if beta_of is not None:
        out["dbeta"] = slope / float(model["beta"])
    return out


def _nu0_A(model, grid, r, v):
    """1e-3 of the mean squared column norm of A, from 64 of the samples."""
    x = _centres(grid)
    pick = torch.linspace(0, r.shape[0] - 1, 64, device=DEV).long()
    B = float(model["beta"]) * torch.tensor(model["G"], dtype=F64, device=DEV)
    X, R, W = x @ B.T, r[pick].double() @ B.T, v[pick].double() @ B.T
    y = X[None] - R[:, None]
    a, d = _scalars((y * y).sum(2))
    J = a[..., None] * W[:, None] + (d * (y * W[:, None]).sum(2))[..., None] * y
    k = J @ torch.tensor(model["p"], dtype=F64, device=DEV).T
    return 1e-3 * float((k * k).sum()) * r.shape[0] / 64 / x.shape[0]


def _trace_kernel(model, grid):
    """beta tr(K(beta G y) G) on all voxel offsets, [2 ny - 1, 2 nx - 1]."""
    B = float(model["beta"]) * torch.tensor(model["G"], dtype=F64, device=DEV)
    j = torch.arange(-(grid["ny"] - 1), grid["ny"], dtype=F64, device=DEV) * grid["dy"]
    i = torch.arange(-(grid["nx"] - 1), grid["nx"], dtype=F64, device=DEV) * grid["dx"]
    y = [B[k, 0] * i[None, :] + B[k, 1] * j[:, None] for k in range(2)]
    a, d = _scalars(y[0] ** 2 + y[1] ** 2)
    By = [sum(y[k] * B[k, m] for k in range(2)) for m in range(2)]
    return a * (B[0, 0] + B[1, 1]) + d * (y[0] * By[0] + y[1] * By[1])


def _dense_A(model, x, r, v):
    """A as a dense [n_ch T, N] matrix."""
    B = float(model["beta"]) * torch.tensor(model["G"], dtype=F64, device=DEV)
    X, R, W = x @ B.T, r @ B.T, v @ B.T
    T, N, n_ch = r.shape[0], x.shape[0], len(model["p"])
    A = torch.empty((n_ch, T, N), dtype=F64, device=DEV)
    step = max(1, (1 << 25) // N)
    for t in range(0, T, step):
        e = slice(t, min(T, t + step))
        y = [X[None, :, i] - R[e, i, None] for i in range(2)]
        a, d = _scalars(y[0] ** 2 + y[1] ** 2)
        f = d * (y[0] * W[e, 0, None] + y[1] * W[e, 1, None])
        J = [a * W[e, i, None] + f * y[i] for i in range(2)]
        for k, p in enumerate(model["p"]):
            A[k, e] = p[0] * J[0] + p[1] * J[1]
    return A.reshape(n_ch * T, N)


def _cg(apply, b, x, steps, tol=None):
    r = b - apply(x)
    p, rr, bn = r.clone(), float(torch.sum(r * r)), math.sqrt(float(torch.sum(b * b)))
    for _ in range(steps):
        if rr == 0.0 or (tol is not None and math.sqrt(rr) <= tol * bn):
            break
        q = apply(p)
        pq = float(torch.sum(p * q))
        if pq == 0.0:
            break
        x = x + (rr / pq) * p
        r = r - (rr / pq) * q
        new = float(torch.sum(r * r))
        p = r + (new / rr) * p
        rr = new
    return x


def _smooth(x):
    """The built-in denoiser: 5-tap Gaussian, mirrored edges, rows then columns."""
    w = torch.exp(-0.5 * torch.arange(-2, 3, dtype=F64, device=DEV) ** 2)
    w = w / w.sum()
    for axis in (1, 0):
        n = x.shape[axis]
        at = torch.arange(n, device=DEV)
        acc = torch.zeros_like(x)
        for m in range(-2, 3):
            i = (at + m) % (2 * n)
            acc += w[m + 2] * x.index_select(axis, torch.where(i >= n, 2 * n - 1 - i, i))
        x = acc
    return x


def _algorithm1(normal, b0, n_iter, n_cg, nu0):
    rho, nu, lam = torch.zeros_like(b0), nu0, 0.0
    for k in range(n_iter):
        x = _cg(lambda q, nu=nu: normal(q) + nu * q, b0 + nu * rho, rho, n_cg)
        srt = x.reshape(-1).sort().values
        h = (srt.numel() - 1) * 0.05
        lo = int(math.floor(h))
        hi = min(lo + 1, srt.numel() - 1)
        x = torch.clamp(x, min=float(srt[lo] + (h - lo) * (srt[hi] - srt[lo])))
        var = float(((x - x.mean()) ** 2).mean())
        lam = nu0 * var if k == 0 else lam
        rho = _smooth(x)
        nu = lam / var if var > 0 else nu
    return rho


def _cell(grid, r):
    """Per axis: lower node and the upper node's cosine weight."""
    out = []
    for k, q in enumerate("xyz"[:r.shape[1]]):
        n = grid["n" + q]
        f = (r[:, k] - grid[q + "0"]) / grid["d" + q] - 0.5
        lo = torch.clamp(torch.floor(f), 0, max(0, n - 2))
        t = torch.clamp(f - lo, 0.0, 1.0)
        out.append((lo.long(), 0.5 * (1 - torch.cos(math.pi * t)) if n > 1 else torch.zeros_like(t)))
    return out


def _core(case, st, tol=None, steps=None, gamma=1e-7, scaled=False):
    grid, r, v, s = st["grid"], st["r"].double(), st["v"].double(), st["s"].double()
    dim, T = r.shape[1], r.shape[0]
    shape = [grid["n" + q] for q in "xyz"[:dim]][::-1]
    N, cells = math.prod(shape), _cell(grid, r)
    stride = [math.prod(shape[dim - k:]) for k in range(dim)]  # x fastest
    corner = []
    for b in range(2 ** dim):
        at, w = torch.zeros(T, dtype=torch.long, device=DEV), torch.ones(T, dtype=F64, device=DEV)
        for k in range(dim):
            up = (b >> k) & 1
            at = at + (cells[k][0] + (up if grid["n" + "xyz"[k]] > 1 else 0)) * stride[k]
            w = w * (cells[k][1] if up else 1 - cells[k][1])
        corner.append((at, w))

    def M(A):
        val = sum(A[:, at] * w for at, w in corner).reshape(dim, dim, T)
        return (val * v.T[None]).sum(1)

    def MT(y):
        wv = (y[:, None, :] * v.T[None]).reshape(dim * dim, T)
        out = torch.zeros((dim * dim, N), dtype=F64, device=DEV)
        for at, w in corner:
            out.index_add_(1, at, wv * w)
        return out

    def lap(A):
        A = A.reshape([-1] + shape)
        out = torch.zeros_like(A)
        for k in range(dim):
            ax, n = dim - k, grid["n" + "xyz"[k]]
            h = 1.0 / grid["d" + "xyz"[k]] ** 2 if scaled else 1.0
            at = torch.arange(n, device=DEV)
            out += h * (A.index_select(ax, torch.clamp(at - 1, min=0)) + A.index_select(ax, torch.clamp(at + 1, max=n - 1))
                        - 2 * A)
        return out.reshape(-1, N)

    A = _cg(lambda x: MT(M(x)) / T + gamma * lap(lap(x)), MT(s) / T,
            torch.zeros((dim * dim, N), dtype=F64, device=DEV), steps or 10000, tol)
    A = A.reshape([-1] + shape)
    return A, sum(A[k * dim + k] for k in range(dim))


def exact(case, seed):
    kind, N, T = case["kind"], _voxels(case), case["T"]
    if kind in ("forward", "adjoint", "normal", "gradient", "pair3") and N * T > 2.2e10:
        return None  # minutes of 64-bit pair sums
    st = prepare(case, seed)
    model, grid, r, v = st["model"], st["grid"], st["r"].double(), st["v"].double()
    if kind in ("core", "core3"):
        A, u = _core(case, st, steps=case["steps"], gamma=case["gamma"], scaled=case["scaled"])
        return {"A": A, "u": u}
    if kind == "two_stage":
        A, u = _core(case, st, tol=1e-3, scaled=True)
        K = _trace_kernel(model, grid)
        ny, nx = grid["ny"], grid["nx"]
        full = (3 * ny - 2, 3 * nx - 2)
        Kf = torch.fft.rfft2(K, full)

        def C(x):
            return torch.fft.irfft2(Kf * torch.fft.rfft2(x, full), full)[ny - 1:2 * ny - 1, nx - 1:2 * nx - 1]
        return {"A": A, "rho": _algorithm1(lambda q: C(C(q)), C(u), case["n_iter"], case["n_cg"], st["nu0"])}
    x = _centres(grid)
    if kind == "recon":
        A = _dense_A(model, x, r, v)
        shape = (grid["ny"], grid["nx"])
        return _algorithm1(lambda q: (A.T @ (A @ q.reshape(-1))).reshape(shape),
                           (A.T @ st["s"].double().reshape(-1)).reshape(shape), case["n_iter"], case["n_cg"], st["nu0"])
    shape = [grid["n" + q] for q in "xyz" if "n" + q in grid][::-1]
    c = st["c"].detach().double().reshape(-1) if "c" in st else None
    if kind == "forward":
        return _sweep(model, x, r, v, c=c)["s"]
    if kind == "adjoint":
        return _sweep(model, x, r, v, s=st["s"].double())["c"].reshape(shape)
    if kind == "pair3":
        got = _sweep(model, x, r, v, c=c, s=st["s"].double())
        return {"s": got["s"], "c": got["c"].reshape(shape)}
    s = _sweep(model, x, r, v, c=c)["s"]
    if kind == "normal":
        return {"s": s, "c": _sweep(model, x, r, v, s=s)["c"].reshape(shape)}
    got = _sweep(model, x, r, v, s=s - st["s"].double(), beta_of=c)
    return {"s": s, "dc": got["c"].reshape(shape), "dbeta": torch.tensor(got["dbeta"], dtype=F64)}
