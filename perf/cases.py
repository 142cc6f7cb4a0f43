"""The calls whose speed this library is judged by, over the sizes it is used at.

Suspensions are seeded random placements at the densities of the library's own workloads: boomerangs of
15 blobs (128 bodies in a 40 um box, scaled with the body count; 256 bodies in a 45.3 um pseudo-periodic
cell) and rollers of 12 blobs, lowest blob at a + Exp(1.5 a) above the wall, forces N(0, 1).  Blob counts
are multiples of 15 or 12, so no size is a multiple of a tile.

Kinds:
  matvec   U = M F through Handle.mobility_apply, FP32 or FP64, k right-hand sides, open or periodic
  batch    U = M F of many uneven suspensions through Handle.mobility_apply_batched
  grad     forward and backward of autograd.mobility_apply (FP64): U, dL/dr, dL/dF
  adjoint  the FP32 position gradient of sum_m u_m^T M F_m
  solve    the saddle-point mobility solve by GMRES with the block preconditioner (FP64 pairs)
  step     one trapezoidal-slip time step (FP32 pairs): Lanczos, three solves, RFD drift

exact() is the textbook Rotne-Prager-Blake mobility in torch float64 (dense rows), torch's autograd for
the gradients and a dense LU for the solve.
"""
import math

import numpy as np
import torch

from paper_1709_02410_gb300 import F32, F64, Forces, Handle, StepParams
from paper_1709_02410_gb300 import autograd

ETA, KT, S_MIN = 1.0e-3, 0.0041, 1.0e-3
RADIUS = {"boomerang": 0.325, "roller": 0.416}
ARM = 14.7 * 0.325  # seven blob spacings of 2.1 a: the boomerang's length scale in the RFD


def listed():
    return [
        # the smallest call: a handful of bodies, as in a test or a parameter scan; launches and latency
        {"name": "matvec-f32-240", "kind": "matvec", "shape": "boomerang", "bodies": 16, "k": 1, "dtype": "f32", "cell": "open"},
        # 128 boomerangs in a 40 um box, one Krylov matvec of a small run
        {"name": "matvec-f32-1920", "kind": "matvec", "shape": "boomerang", "bodies": 128, "k": 1, "dtype": "f32", "cell": "open"},
        # the large suspension's Krylov matvec: most of a production time step
        {"name": "matvec-f32-65535", "kind": "matvec", "shape": "boomerang", "bodies": 4369, "k": 1, "dtype": "f32", "cell": "open"},
        # many force fields on one configuration (mobility statistics): 16 right-hand sides at once
        {"name": "matvec-f32-k16-65535", "kind": "matvec", "shape": "boomerang", "bodies": 4369, "k": 16, "dtype": "f32", "cell": "open"},
        # the paper's own suspension, 256 boomerangs in a periodic cell: nine images a pair
        {"name": "matvec-f32-periodic-3840", "kind": "matvec", "shape": "boomerang", "bodies": 256, "k": 1, "dtype": "f32", "cell": "periodic"},
        # reference-precision matvec, what float64 tensors get by default
        {"name": "matvec-f64-1920", "kind": "matvec", "shape": "boomerang", "bodies": 128, "k": 1, "dtype": "f64", "cell": "open"},
        # 64 independent suspensions of 480 to 22,500 blobs in one call
        {"name": "batch-f32-64", "kind": "batch", "systems": 64, "least": 32, "most": 1500, "layout": 4, "k": 1},
        # differentiable mobility: a loss on the velocities, gradients to positions and forces
        {"name": "grad-f64-1920", "kind": "grad", "shape": "boomerang", "bodies": 128},
        # position gradient at the adjoint's working size
        {"name": "adjoint-f32-16380", "kind": "adjoint", "shape": "boomerang", "bodies": 1092, "k": 1},
        # deterministic mobility problem of 128 bodies, solved in the default precision
        {"name": "solve-f64-1920", "kind": "solve", "shape": "boomerang", "bodies": 128, "tol": 1e-6},
        # a time step of the paper's periodic suspension at the paper's solver tolerances
        {"name": "step-f32-periodic-3840", "kind": "step", "bodies": 256, "cell": "periodic", "tol": 1e-3, "tol_lanczos": 1e-3},
        # the production step: 65,535 blobs at the tight tolerances of the library's benchmark
        {"name": "step-f32-65535", "kind": "step", "bodies": 4369, "cell": "open", "tol": 1e-6, "tol_lanczos": 1e-4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "matvec", "periodic", "f64", "batch", "grad", "adjoint", "solve", "step"])
    shape = rng.choice(["boomerang", "boomerang", "roller"])
    if kind == "matvec":
        k = rng.choice([1, 1, 2, 4, 16, rng.randint(1, 16)])
        return {"kind": "matvec", "shape": shape, "bodies": _log_int(rng, 2, 4369), "k": k, "dtype": "f32", "cell": "open"}
    if kind == "periodic":
        return {"kind": "matvec", "shape": "boomerang", "bodies": _log_int(rng, 16, 1024), "k": rng.choice([1, 1, 2]),
                "dtype": "f32", "cell": "periodic"}
    if kind == "f64":
        return {"kind": "matvec", "shape": shape, "bodies": _log_int(rng, 4, 512), "k": rng.choice([1, 1, 2, 4]), "dtype": "f64",
                "cell": rng.choice(["open", "open", "periodic"])}
    if kind == "batch":
        least = _log_int(rng, 8, 64)
        return {"kind": "batch", "systems": rng.randint(5, 64), "least": least, "most": _log_int(rng, 128, 1500),
                "layout": rng.randrange(1 << 20), "k": rng.choice([1, 1, 2, 4])}
    if kind == "grad":
        return {"kind": "grad", "shape": shape, "bodies": _log_int(rng, 4, 256)}
    if kind == "adjoint":
        return {"kind": "adjoint", "shape": shape, "bodies": _log_int(rng, 16, 1092), "k": rng.choice([1, 1, 2, 3, 4])}
    if kind == "solve":
        return {"kind": "solve", "shape": shape, "bodies": _log_int(rng, 8, 256), "tol": rng.choice([1e-4, 1e-6, 1e-8])}
    return {"kind": "step", "bodies": _log_int(rng, 16, 1024), "cell": rng.choice(["open", "periodic"]), "tol": 1e-3,
            "tol_lanczos": 1e-3}


# ---- inputs ----------------------------------------------------------------


def _reference(shape):
    """Blob offsets of one body, [nper, 3]."""
    a = RADIUS[shape]
    if shape == "boomerang":
        s = np.zeros((15, 3))
        s[1:8, 0] = s[8:15, 1] = 2.1 * a * np.arange(1, 8)
        return s
    g = (1 + 5 ** 0.5) / 2
    return a * np.array([p for u in (-1, 1) for v in (-1, 1) for p in ((0, u, v * g), (u, v * g, 0), (v * g, 0, u))], dtype=float)


def _side(shape, bodies, cell="open"):
    """Edge of the square the body centres are placed in (um)."""
    if cell == "periodic":
        return 45.3 * math.sqrt(bodies / 256)
    if shape == "roller":
        return math.sqrt(bodies * math.pi * 0.656 ** 2 / 0.4)
    return 40.0 * math.sqrt(bodies / 128)


def _bodies(rng, shape, bodies, cell="open"):
    """Tracking points [nb, 3], unit quaternions [nb, 4] and blob positions [3, n]."""
    a, s = RADIUS[shape], _reference(shape)
    q = np.empty((bodies, 3))
    q[:, :2] = rng.uniform(0, _side(shape, bodies, cell), (bodies, 2))
    th = rng.standard_normal((bodies, 4))
    th /= np.linalg.norm(th, axis=1, keepdims=True)
    w, x, y, z = th.T
    R = np.stack([w * w + x * x - y * y - z * z, 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), w * w - x * x + y * y - z * z, 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), w * w - x * x - y * y + z * z], 1).reshape(bodies, 3, 3)
    d = np.einsum("bij,kj->bki", R, s)
    q[:, 2] = a + rng.exponential(1.5 * a, bodies) - d[:, :, 2].min(axis=1)
    return q, th, np.ascontiguousarray((q[:, None, :] + d).reshape(-1, 3).T)


def _counts(case):
    """Body count of every system of a batch (log-uniform), fixed by the case's layout."""
    lo, hi = sorted((case["least"], case["most"]))
    u = np.random.default_rng(case["layout"]).uniform(math.log(lo), math.log(hi), case["systems"])
    return np.floor(np.exp(u)).astype(int)


def _make(case, seed):
    """The case's inputs as numpy arrays, from the seed alone."""
    rng = np.random.default_rng([seed, 17])
    if case["kind"] == "batch":
        counts = _counts(case)
        r = np.concatenate([_bodies(rng, "boomerang", int(c))[2] for c in counts], axis=1)
        off = np.concatenate([[0], np.cumsum(15 * counts)]).astype(np.int64)
        return {"r": r, "off": off, "F": rng.standard_normal((case["k"], 3, r.shape[1]), dtype=np.float32)}
    q, th, r = _bodies(rng, case.get("shape", "boomerang"), case["bodies"], case.get("cell", "open"))
    n, nb = r.shape[1], case["bodies"]
    if case["kind"] == "matvec":
        shp = (3, n) if case["k"] == 1 else (case["k"], 3, n)
        return {"r": r, "F": rng.standard_normal(shp, dtype=np.float32 if case["dtype"] == "f32" else np.float64)}
    if case["kind"] == "grad":
        return {"r": r, "F": rng.standard_normal((3, n)), "G": rng.standard_normal((3, n))}
    if case["kind"] == "adjoint":
        shp = (3, n) if case["k"] == 1 else (case["k"], 3, n)
        return {"r": r, "u": rng.standard_normal(shp), "F": rng.standard_normal(shp)}
    if case["kind"] == "solve":
        return {"r": r, "q": q, "slip": rng.standard_normal((3, n)), "FT": 1e-2 * rng.standard_normal((nb, 6))}
    return {"q": q, "theta": th}


def _handle(case):
    L = _side("boomerang", case["bodies"], "periodic") if case.get("cell") == "periodic" else 0.0
    return Handle(ETA, RADIUS[case.get("shape", "boomerang")], KT, wall=True, s_min=S_MIN, Lx=L, Ly=L)


def prepare(case, seed):
    x = _make(case, seed)
    s = {"kind": case["kind"], "h": _handle(case)}
    for name, v in x.items():
        s[name] = v if name == "off" else torch.from_numpy(v).to("cuda")
    if case["kind"] == "grad":
        s["r"].requires_grad_()
        s["F"].requires_grad_()
    if case["kind"] == "solve":
        s["nper"], s["tol"] = _reference(case["shape"]).shape[0], case["tol"]
    if case["kind"] == "step":
        s["shape"] = torch.from_numpy(_reference("boomerang")).to("cuda")
        # gravity and wall repulsion of the library's benchmark step
        s["forces"] = Forces(1.57e-11 * 9.81e6, 0.096, 0.162, 0.1, (0.0, 0.0, 0.0))
        s["sp"] = StepParams(0.01, 1e-3, ARM, case["tol"], case["tol_lanczos"], 300, 100, 80, F32, seed, 0)
    return s


# ---- one pass --------------------------------------------------------------


def run(s):
    h, kind = s["h"], s["kind"]
    if kind == "matvec":
        return h.mobility_apply(s["r"], s["F"])
    if kind == "batch":
        return h.mobility_apply_batched(s["off"], s["r"], s["F"])
    if kind == "grad":
        U = autograd.mobility_apply(h, s["r"], s["F"])
        gr, gF = torch.autograd.grad(U, (s["r"], s["F"]), s["G"])
        return {"U": U, "gr": gr, "gF": gF}
    if kind == "adjoint":
        # the gradient of an FP32 evaluation, handed on in FP32
        return h.mobility_adjoint(s["r"], s["u"], s["F"], dtype=F32).float()
    if kind == "solve":
        lam, U, _ = h.gmres_rigid_solve(s["nper"], s["r"], s["q"], s["slip"], s["FT"], tol=s["tol"], max_iter=300, restart=100,
                                        dtype=F64)
        return {"lambda": lam, "U": U}
    # the step advances q and theta in place: each pass from the state's own configuration; the frame is
    # kept in FP32, the precision of the step's pair arithmetic
    q, theta = s["q"].clone(), s["theta"].clone()
    h.step_ts(s["shape"], q, theta, s["forces"], s["sp"])
    return {"q": q.float(), "theta": theta.float()}


# ---- what a pass cannot do without ------------------------------------------


def work(case):
    """Flops: one block per unordered pair (67 for its scalars, nine images in the periodic cell) and 18 per
    right-hand side for each of its two directions; gradients: the block's scalars with three derivatives
    (4 x) and two contractions.  Solves and steps: the matvecs they need (typical iteration counts)."""
    kind = case["kind"]
    if kind == "batch":
        n = 15.0 * _counts(case)
        return {"bytes": float(n.sum()) * (24 + 24 * case["k"]), "flops": float((n * n).sum()) * (33.5 + 18 * case["k"])}
    n = float(case["bodies"] * (12 if case.get("shape") == "roller" else 15))
    images = 9 if case.get("cell") == "periodic" else 1
    k = case.get("k", 1)
    pair = images * (33.5 + 18 * k)
    if kind == "matvec":
        return {"bytes": n * (24 + 6 * k * (4 if case["dtype"] == "f32" else 8)), "flops": n * n * pair}
    if kind == "grad":
        return {"bytes": n * 6 * 24, "flops": n * n * (2 * 51.5 + 134 + 70)}
    if kind == "adjoint":
        return {"bytes": n * (24 + 48 * k + 24), "flops": n * n * (134 + 70 * k)}
    if kind == "solve":
        return {"bytes": n * 24 * 4, "flops": 35 * n * n * pair}
    return {"bytes": n * 24 * 4, "flops": (115 if case["tol"] < 1e-4 else 60) * n * n * pair}


# ---- the same results in plain 64-bit torch ----------------------------------


def _clamped(r, a):
    """Heights clamped to the blob radius and the overlap scale of every blob."""
    return torch.stack([r[0], r[1], r[2].clamp(min=a)]), (r[2] / a).clamp(S_MIN, 1.0)


def _block(ri, rj, a, L):
    """8 pi eta M of targets ri [3, m] and sources rj [3, n]: entries [3][3] of [m, n] matrices (Rotne-Prager
    in free space plus Blake's images with the Faxen corrections of both blobs), summed over the minimum
    image and its eight neighbours when L > 0."""
    x0, y0 = ri[0][:, None] - rj[0][None], ri[1][:, None] - rj[1][None]
    dz, zj = ri[2][:, None] - rj[2][None], rj[2][None]
    Rz = ri[2][:, None] + zj
    if L > 0:
        x0, y0 = x0 - L * torch.round(x0.detach() / L), y0 - L * torch.round(y0.detach() / L)
    M = [[0.0] * 3 for _ in range(3)]
    shifts = [(u * L, v * L) for u in (-1, 0, 1) for v in (-1, 0, 1)] if L > 0 else [(0.0, 0.0)]
    for sx, sy in shifts:
        d = (x0 + sx, y0 + sy, dz)
        rho2 = d[0] * d[0] + d[1] * d[1]
        r2 = rho2 + dz * dz
        own = r2 == 0
        r2 = torch.where(own, torch.ones_like(r2), r2)
        r = r2.sqrt()
        near = r < 2 * a
        c1 = torch.where(near, 4 / (3 * a) * (1 - 9 * r / (32 * a)), (1 + 2 * a * a / (3 * r2)) / r)
        c2 = torch.where(near, 1 / (8 * a * a * r), (1 - 2 * a * a / r2) / (r2 * r))
        c1 = torch.where(own, torch.full_like(c1, 4 / (3 * a)), c1)
        c2 = torch.where(own, torch.zeros_like(c2), c2)
        R = (rho2 + Rz * Rz).sqrt()
        ez, t, s2 = Rz / R, zj / R, (a / R) ** 2
        e2, s4 = ez * ez, s2 * s2
        A = -1 - 2 * ez * t + 2 * t * t + s2 * (2 * e2 - 2 / 3) + s4 * (2 / 3 - 10 / 3 * e2)
        B = -1 + 6 * ez * t - 6 * t * t + s2 * (2 - 10 * e2) + s4 * (70 / 3 * e2 - 10 / 3)
        C = t * (2 - 12 * e2) + 12 * ez * t * t + ez * s2 * (20 * e2 - 4) + ez * s4 * (40 / 3 - 140 / 3 * e2)
        D = 2 * t - 20 / 3 * ez * s4
        E = -4 * t * t - 4 * e2 * s2 + s4 * (20 * e2 - 8 / 3)
        e = (d[0] / R, d[1] / R, ez)
        for i in range(3):
            for j in range(3):
                m = c2 * d[i] * d[j] + B / R * e[i] * e[j]
                if i == j:
                    m = m + c1 + A / R
                if j == 2:
                    m = m + C / R * e[i]
                if i == 2:
                    m = m + D / R * e[j]
                if i == 2 and j == 2:
                    m = m + E / R
                M[i][j] = M[i][j] + m
    return M


def _rows(n, images=1, per=30e6):
    return max(1, min(n, int(per / (n * (1 if images == 1 else 2)))))


def _apply(r, F, a, L=0.0):
    """M F in float64, [k, 3, n] forces, target rows in chunks."""
    rt, s = _clamped(r, a)
    f = F * s
    n, U = r.shape[1], torch.empty_like(F)
    step = _rows(n, 9 if L > 0 else 1)
    for i in range(0, n, step):
        M = _block(rt[:, i:i + step], rt, a, L)
        for c in range(3):
            U[:, c, i:i + step] = sum(f[:, d] @ M[c][d].T for d in range(3)) * s[i:i + step]
    return U / (8 * math.pi * ETA)


def _gradient(r, u, F, a):
    """d(sum_m u_m^T M F_m)/dr by autograd, target rows in chunks."""
    n, g = r.shape[1], torch.zeros_like(r)
    step = _rows(n, per=8e6)
    for i in range(0, n, step):
        x = r.detach().clone().requires_grad_()
        rt, s = _clamped(x, a)
        M = _block(rt[:, i:i + step], rt, a, 0.0)
        us, fs = u[:, :, i:i + step] * s[i:i + step], F * s
        e = sum((us[m, c] * (M[c][d] @ fs[m, d])).sum() for m in range(u.shape[0]) for c in range(3) for d in range(3))
        g += torch.autograd.grad(e, x)[0]
    return g / (8 * math.pi * ETA)


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None
    x = {k: v if k == "off" else torch.from_numpy(v).to("cuda", torch.float64) for k, v in _make(case, seed).items()}
    a = RADIUS[case.get("shape", "boomerang")]
    L = _side("boomerang", case["bodies"], "periodic") if case.get("cell") == "periodic" else 0.0
    if kind == "matvec":
        F = x["F"] if x["F"].dim() == 3 else x["F"][None]
        return _apply(x["r"], F, a, L).reshape(x["F"].shape)
    if kind == "batch":
        off = x["off"]
        return torch.cat([_apply(x["r"][:, i:j].contiguous(), x["F"][:, :, i:j].contiguous(), a) for i, j in zip(off, off[1:])], dim=2)
    if kind == "grad":
        return {"U": _apply(x["r"], x["F"][None], a)[0], "gr": _gradient(x["r"], x["G"][None], x["F"][None], a),
                "gF": _apply(x["r"], x["G"][None], a)[0]}
    if kind == "adjoint":
        u, F = (v if v.dim() == 3 else v[None] for v in (x["u"], x["F"]))
        return _gradient(x["r"], u, F, a)
    # solve: [M -K; -K^T 0] [lambda; U] = [-slip; -FT], rows c * n + i
    r, q, nb = x["r"], x["q"], case["bodies"]
    n = r.shape[1]
    rt, s = _clamped(r, a)
    blocks = _block(rt, rt, a, 0.0)
    A = torch.zeros((3 * n + 6 * nb, 3 * n + 6 * nb), dtype=torch.float64, device="cuda")
    for c in range(3):
        for d in range(3):
            A[c * n:(c + 1) * n, d * n:(d + 1) * n] = s[:, None] * blocks[c][d] * s[None] / (8 * math.pi * ETA)
    p = torch.arange(nb, device="cuda").repeat_interleave(n // nb)
    i = torch.arange(n, device="cuda")
    o = r - q.T[:, p]
    K = torch.zeros((3 * n, 6 * nb), dtype=torch.float64, device="cuda")
    for c in range(3):
        K[c * n + i, 6 * p + c] = 1.0
        b, d = (c + 1) % 3, (c + 2) % 3  # (omega x o)_c = omega_b o_d - omega_d o_b
        K[c * n + i, 6 * p + 3 + b] = o[d]
        K[c * n + i, 6 * p + 3 + d] = -o[b]
    A[:3 * n, 3 * n:] = -K
    A[3 * n:, :3 * n] = -K.T
    b = torch.cat([-x["slip"].reshape(-1), -x["FT"].reshape(-1)])
    y = torch.linalg.solve(A, b)
    return {"lambda": y[:3 * n].reshape(3, n), "U": y[3 * n:].reshape(nb, 6)}
