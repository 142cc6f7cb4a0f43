"""Pair kernels at the edges of their tiles: one blob more or less than a warp,
a home tile or the size at which the work is cut differently, against the
oracle (the tolerances of each precision: 1e-5 in FP32, 1e-12 in FP64)."""
import numpy as np
import pytest
import torch

from oracle import mobility as om, saddle
from paper_1709_02410_gb300 import F32, F64, Handle, synth

from gpu_util import rel2, to_dev

pytestmark = pytest.mark.gpu

CELL = 45.3


def cloud(n, seed, side=None):
    """n blobs at the boomerang suspensions' density, overlapping pairs and blobs below the wall height a among them."""
    rng = np.random.default_rng(seed)
    a = synth.A_BOOMERANG
    side = 40.0 * np.sqrt(max(n, 60) / 1920) if side is None else side
    r = np.empty((3, n))
    r[:2] = rng.uniform(0.0, side, (2, n))
    r[2] = 0.7 * a + rng.exponential(3.0 * a, n)
    return r


def rows_of(n):
    """Sampled target blobs: all of a small system, else the tile edges and some between."""
    if n <= 600:
        return np.arange(n)
    e = np.array([0, 31, 32, 63, 64, 127, 128, 255, 256, n - 257, n - 256, n - 33, n - 32, n - 1])
    return np.unique(np.concatenate([e, np.linspace(0, n - 1, 40).astype(int)]))


# 8,704 = 34 home tiles of 256: the last size with one visitor tile per item; variant 3: those kernels below
# 960 blobs too, where the default is one launch (640 with three or four right-hand sides)
@pytest.mark.parametrize("n,variant", [(n, v) for v in (-1, 3) for n in (1, 2, 31, 33, 64, 255, 257, 513, 8704, 8993)
                                       if v == -1 or n < 8000] + [(n, -1) for n in (304, 305, 609, 640, 641, 960, 961)])
@pytest.mark.parametrize("cell", [0.0, CELL])
def test_f32_symmetric_tiles(n, variant, cell):
    r = cloud(n, 700 + n, cell or None)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT, Lx=cell, Ly=cell)
    h.set_sym_variant(variant)
    prm = om.Params(synth.ETA, synth.A_BOOMERANG, Lx=cell, Ly=cell)
    rows = rows_of(n)
    for k in (1, 2, 3):
        F = synth.gaussian(701 + k, (k, 3, n), np.float32)
        U = h.mobility_apply(to_dev(r), to_dev(F, torch.float32)).cpu().numpy()
        assert rel2(U[:, :, rows], om.apply(r, F.astype(np.float64), prm, rows)) <= 1e-5


# (the last: items of several visitor tiles, four homes per thread)
@pytest.mark.parametrize("sizes", [(1, 255, 256, 257), (33, 513, 64), (300,) * 40, (6000, 12, 7001)])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_f32_symmetric_batches(sizes, k):
    """Batches of short items, two home blobs per thread, and of longer ones, four, each system against the oracle."""
    rs = [cloud(n, 770 + i) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
    h.set_batch_variant(4)
    prm = om.Params(synth.ETA, synth.A_BOOMERANG)
    F = synth.gaussian(771, (k, 3, off[-1]), np.float32)
    U = h.mobility_apply_batched(off, to_dev(np.concatenate(rs, axis=1)), to_dev(F, torch.float32)).cpu().numpy()
    for s, r in enumerate(rs):
        sl, rows = slice(off[s], off[s + 1]), rows_of(r.shape[1])
        assert rel2(U[:, :, sl][:, :, rows], om.apply(r, F[:, :, sl].astype(np.float64), prm, rows)) <= 1e-5


def test_accumulators_are_cleared_between_calls():
    """One handle, calls of other sizes, right-hand sides and a non-finite force between: every result as on a fresh handle."""
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
    h.set_sym_variant(3)  # (small systems default to a kernel without accumulators)
    for n, k, bad in ((700, 2, False), (300, 1, True), (300, 1, False), (1100, 4, False), (40, 1, False), (700, 2, False)):
        r, F = cloud(n, 710), synth.gaussian(711, (k, 3, n), np.float32)
        if bad:
            F[0, 1, 7] = np.inf
        args = to_dev(r), to_dev(F, torch.float32)
        U = h.mobility_apply(*args)
        g = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
        g.set_sym_variant(3)
        fresh = g.mobility_apply(*args)
        assert torch.isnan(U).all() if bad else torch.equal(U, fresh)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_nan_position_gives_nan(dtype):
    """A NaN coordinate, the height too (clamped, but its overlap scale is NaN), shows in U."""
    for c in range(3):
        r, F = cloud(300, 720), synth.gaussian(721, (3, 300))
        r[c, 40] = np.nan
        U = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT).mobility_apply(to_dev(r), to_dev(F, dtype))
        assert torch.isnan(U[:, 40]).all()


# 4,096 / 4,097: one and four warps per CTA
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 65, 255, 1937, 4096, 4097, 4225])
@pytest.mark.parametrize("wall,cell", [(True, 0.0), (True, CELL), (False, 0.0)])
def test_f64_symmetric_tiles(n, wall, cell):
    r = cloud(n, 730 + n, cell or None)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT, wall=wall, Lx=cell, Ly=cell)
    prm = om.Params(synth.ETA, synth.A_BOOMERANG, wall=wall, Lx=cell, Ly=cell)
    rows = rows_of(n)
    for k in (1, 2, 3) if n > 600 else (1, 2, 4, 7, 9):
        F = synth.gaussian(731 + k, (k, 3, n))
        U = h.mobility_apply(to_dev(r), to_dev(F)).cpu().numpy()
        assert rel2(U[:, :, rows], om.apply(r, F, prm, rows)) <= 1e-12


# FP64: 32 homes a warp, four warps past 4,096; FP32: 64 homes a warp, four warps past 8,192
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 65, 255, 1937, 4097, 8193])
@pytest.mark.parametrize("wall,cell", [(True, 0.0), (True, CELL), (False, 0.0)])
def test_adjoint_tiles(n, wall, cell):
    r = cloud(n, 740 + n, cell or None)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT, wall=wall, Lx=cell, Ly=cell)
    prm = om.Params(synth.ETA, synth.A_BOOMERANG, wall=wall, Lx=cell, Ly=cell)
    rows = rows_of(n)
    for k in (1,) if n > 600 else (1, 2, 3, 6):
        u, F = synth.gaussian(741 + k, (2, k, 3, n))
        go = sum(om.grad(r, u[m], F[m], prm, rows) for m in range(k))
        for dtype, tol in ((F64, 1e-11), (F32, 1e-5)):
            g = h.mobility_adjoint(to_dev(r), to_dev(u), to_dev(F), dtype=dtype).cpu().numpy()
            assert np.linalg.norm(g[:, rows] - go) <= tol * np.linalg.norm(go)  # (a lone unbounded blob has none)


# two targets per thread (256 a CTA), 64 sources a stage
@pytest.mark.parametrize("n", [1, 63, 65, 128, 129, 257, 2113])
@pytest.mark.parametrize("cell", [0.0, CELL])
def test_f32_many_right_hand_sides(n, cell):
    r = cloud(n, 750 + n, cell or None)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT, Lx=cell, Ly=cell)
    prm = om.Params(synth.ETA, synth.A_BOOMERANG, Lx=cell, Ly=cell)
    rows = rows_of(n)
    for k in (5, 8, 9, 16):
        F = synth.gaussian(751 + k, (k, 3, n), np.float32)
        ref = om.apply(r, F.astype(np.float64), prm, rows)
        for partials in (False, True):
            h.set_sym_partials(partials)
            U = h.mobility_apply(to_dev(r), to_dev(F, torch.float32)).cpu().numpy()
            assert rel2(U[:, :, rows], ref) <= 1e-5


def test_small_system_non_finite_force():
    """A force that is not finite makes every velocity NaN, as with the accumulators of larger systems."""
    r, F = cloud(200, 760), synth.gaussian(761, (2, 3, 200), np.float32)
    F[1, 2, 11] = np.inf
    U = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT).mobility_apply(to_dev(r), to_dev(F, torch.float32))
    assert torch.isnan(U).all()


@pytest.mark.parametrize("dtype,n,tol", [(F32, 217_001, 1e-5), (F64, 127_003, 1e-11)])
def test_adjoint_in_groups(dtype, n, tol):
    """Past the partials' bound the home tiles run in several launches whose sums are carried over."""
    r = cloud(n, 770)
    u, F = synth.gaussian(771, (2, 3, n))
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
    rows = rows_of(n)
    before = h.lib.rpbd_launch_count()
    g = h.mobility_adjoint(to_dev(r), to_dev(u), to_dev(F), dtype=dtype).cpu().numpy()
    assert h.lib.rpbd_launch_count() - before > (1 if dtype == F64 else 3)  # more than one group
    assert rel2(g[:, rows], om.grad(r, u, F, om.Params(synth.ETA, synth.A_BOOMERANG), rows)) <= tol


@pytest.mark.parametrize("nper", [3, 8, 9, 16, 17, 32])
def test_saddle_solve_by_blobs_per_body(nper):
    """Bodies of 3 to 32 blobs (8, 16 or 32 lanes of a warp each, an odd number of bodies) against the dense solution."""
    a = synth.A_BOOMERANG
    L = np.zeros((nper, 3))
    L[:, 0] = np.maximum(nper // 2 - np.arange(nper), 0)  # one arm along x, one along y
    L[:, 1] = np.maximum(np.arange(nper) - nper // 2, 0)
    rng = np.random.default_rng(780 + nper)
    q = np.stack([40.0 * a * np.arange(5), rng.uniform(0, 9 * a, 5), a * rng.uniform(1.5, 4.0, 5)], 1)
    r = (q[:, None] + 2.1 * a * L).reshape(-1, 3).T.copy()
    slip, FT = rng.standard_normal(r.shape), rng.standard_normal((5, 6)) * 1e-2
    prm = om.Params(synth.ETA, a)
    lam_d, U_d, _ = saddle.dense_solution(r, q, nper, prm, slip, FT)
    h = Handle(synth.ETA, a, synth.KT)
    lam, U, st = h.gmres_rigid_solve(nper, to_dev(r), to_dev(q), to_dev(slip), to_dev(FT), tol=1e-12, max_iter=200)
    assert st["status"] == 0
    assert rel2(U.cpu().numpy(), U_d) <= 1e-9 and rel2(lam.cpu().numpy(), lam_d) <= 1e-8


@pytest.mark.parametrize("gap", [1.0, 1e-3, 1e-5, 1e-7, 1e-10])
def test_lanczos_root_by_condition(gap):
    """Two blobs a distance gap a apart (the smallest eigenvalue is proportional to it) among four others, run to the
    full space: 32 quadrature nodes, 64, and the diagonalisation.  Rounding of M moves the root by ~1e-16 sqrt(condition)."""
    a = synth.A_BOOMERANG
    r = a * np.array([[0, 0, 2], [gap, 0, 2], [3, 1, 3], [0, 4, 2.5], [5, 5, 4], [-3, 2, 2]], float).T
    W = synth.gaussian(790, r.shape)
    lam, Q = np.linalg.eigh(om.dense(r, om.Params(synth.ETA, a)))
    ref = om.blob_to_soa(Q @ (np.sqrt(np.maximum(lam, 0)) * (Q.T @ om.soa_to_blob(W))))
    h = Handle(synth.ETA, a, synth.KT)
    out, _ = h.lanczos_sqrt_apply(to_dev(r), to_dev(W), tol=1e-14, max_iter=18, use_precond=False)
    assert rel2(out.cpu().numpy(), ref) <= 1e-9


@pytest.mark.parametrize("sizes", [(1, 127, 0, 128, 129), (385, 2), (40_000, 129, 3)])
def test_batched_lanczos_chunks(sizes):
    """Systems at the edges of the vector kernels' chunks (128 blobs here, 256 in the last case), a fixed number of
    iterations, against one Lanczos per system; FP32 pairs, the tolerance of the batched oracle tests."""
    rs = [cloud(n, 800 + i) for i, n in enumerate(sizes) if n]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    h = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
    W = synth.gaussian(801, (3, off[-1]))
    out, _, it = h.lanczos_sqrt_apply_batched(off, to_dev(np.concatenate(rs, axis=1)), to_dev(W), tol=1e-30, max_iter=7,
                                              use_precond=False)
    g = Handle(synth.ETA, synth.A_BOOMERANG, synth.KT)
    for s, r in zip([s for s, n in enumerate(sizes) if n], rs):
        if r.shape[1] == 1:
            continue  # (three unknowns: the space is exhausted before the seventh iteration)
        Ws = to_dev(np.ascontiguousarray(W[:, off[s]:off[s + 1]]))
        ref, _ = g.lanczos_sqrt_apply(to_dev(r), Ws, tol=1e-30, max_iter=7, dtype=F32, use_precond=False)
        assert it[s] == 7 or r.shape[1] < 3
        assert rel2(out[:, off[s]:off[s + 1]].cpu().numpy(), ref.cpu().numpy()) <= 1e-4
    assert torch.isfinite(out).all()
