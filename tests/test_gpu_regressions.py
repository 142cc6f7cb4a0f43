"""Calls that once went wrong: each test states what it was."""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest
import torch

from oracle import mobility as om
from paper_1709_02410_gb300 import F32, F64, Handle, synth
from paper_1709_02410_gb300.api import RpbdError

from gpu_util import to_dev

pytestmark = pytest.mark.gpu

A = synth.A_BOOMERANG


def cloud(n, seed):
    """n blobs at the boomerang suspensions' density, overlapping pairs and blobs below the wall height a among them."""
    rng = np.random.default_rng(seed)
    r = np.empty((3, n))
    r[:2] = rng.uniform(0.0, 40.0 * np.sqrt(max(n, 60) / 1920), (2, n))
    r[2] = 0.7 * A + rng.exponential(3.0 * A, n)
    return r


def lanczos_batched(h, off, r, W, out, use_graph, stream, iters=None):
    """The C entry; without iters it returns while its work is queued."""
    return h.lib.rpbd_lanczos_sqrt_apply_batched(h.h, off.size - 1, off.ctypes.data_as(C.c_void_p), C.c_void_p(r.data_ptr()),
                                                 C.c_void_p(W.data_ptr()), C.c_void_p(out.data_ptr()), None, None, 1e-30, 7, 0,
                                                 use_graph, iters, C.c_void_p(stream.cuda_stream))


@pytest.mark.parametrize("use_graph", [0, 1])
def test_batched_lanczos_layouts_in_flight(use_graph):
    """Calls with other offsets queued behind one another on a stream of their own: one call's chunk table was written
    over by the next call's while it was read."""
    h = Handle(synth.ETA, A, synth.KT)
    layouts = [np.concatenate([[0], np.cumsum(s)]).astype(np.int64) for s in ((9000, 1, 20_000, 3001), (700,) * 40, (31, 25_000))]
    st = torch.cuda.Stream()
    calls = []
    for i, off in enumerate(layouts):
        n = int(off[-1])
        r, W = to_dev(cloud(n, 900 + i)), to_dev(synth.gaussian(910 + i, (3, n)))
        ref = torch.empty_like(W)
        torch.cuda.synchronize()
        iters = (C.c_int * (off.size - 1))()
        assert lanczos_batched(h, off, r, W, ref, use_graph, st, iters) == 0  # waits; workspaces and graphs exist from here on
        calls.append((off, r, W, ref))
    outs = []
    for off, r, W, ref in calls + calls[::-1]:
        outs.append((torch.zeros_like(W), ref))
    torch.cuda.synchronize()
    for (off, r, W, _), (out, _) in zip(calls + calls[::-1], outs):
        assert lanczos_batched(h, off, r, W, out, use_graph, st) == 0
    st.synchronize()
    for out, ref in outs:
        assert torch.equal(out, ref)


def test_batched_lanczos_refuses_offsets():
    """Offsets that decrease or do not start at 0 are refused before anything is launched: chunks beyond the last
    offset were cut from them."""
    h = Handle(synth.ETA, A, synth.KT)
    r, W = to_dev(cloud(40, 920)), to_dev(synth.gaussian(921, (3, 40)))
    out = torch.full_like(W, 5.0)
    before = h.lib.rpbd_launch_count()
    for off in ((0, 60, 40), (0, 40, 30, 40), (5, 40), (0, -1, 40)):
        assert lanczos_batched(h, np.array(off, np.int64), r, W, out, 0, torch.cuda.current_stream()) == -1
    assert h.lib.rpbd_launch_count() == before and (out == 5.0).all()


# 960 / 961: one launch, three launches (FP32, k <= 2); FP64 k = 6: two passes
@pytest.mark.parametrize("n", [33, 960, 961, 2000])
@pytest.mark.parametrize("cell", [0.0, 45.3])
def test_matvec_in_place(n, cell):
    """U over F, over the positions, and shifted against F by one right-hand side: the one-launch kernel read forces that
    other blocks had overwritten, and later passes of an FP64 matvec read what the first had written."""
    h = Handle(synth.ETA, A, synth.KT, Lx=cell, Ly=cell)
    r = to_dev(cloud(n, 930 + n))
    for dtype, mode in ((torch.float32, None), (torch.float64, None), (torch.float64, F32)):
        for k in (1, 2, 4, 6):
            F = to_dev(synth.gaussian(931 + k, (k, 3, n)), dtype)
            tol = 1e-12 if dtype == torch.float64 and mode is None else 1e-5  # (the other kernel's rounding)
            ref = h.mobility_apply(r, F, dtype=mode)
            near = lambda U: float((U - ref).norm() / ref.norm()) <= tol
            for _ in range(3):
                G = F.clone()
                assert h.mobility_apply(r, G, dtype=mode, out=G) is G and near(G)
                B = torch.zeros((k + 1, 3, n), dtype=dtype, device=r.device)
                B[:k] = F
                assert near(h.mobility_apply(r, B[:k], dtype=mode, out=B[1:]))
                if dtype == torch.float64:
                    B[0] = r
                    assert near(h.mobility_apply(B[0], F, dtype=mode, out=B[:k]))


@pytest.mark.parametrize("k", [1, 2, 4])
def test_small_system_sum_keeps_64_bits(k):
    """Two forces of 1e4 from mirrored places cancel exactly in the velocity along their axis, so what the forces of
    order one leave there has the usual relative error.  (One source a lane; the lanes' sums were added in FP32, which
    loses 2^-24 of the large terms, about 1e-3 here.)"""
    n = 256
    r, F = cloud(n, 940), synth.gaussian(941, (k, 3, n))
    r[:, 0] = 0.0, 0.0, 5.0 * A
    r[:, 17], r[:, 200] = (4.0 * A, 0.0, 3.0 * A), (-4.0 * A, 0.0, 3.0 * A)
    r[:2, 1:17] += 20.0 * A
    F[:, :, 17], F[:, :, 200] = np.array([1e4, 0, 0]), np.array([-1e4, 0, 0])
    F = F.astype(np.float32)
    U = Handle(synth.ETA, A, synth.KT).mobility_apply(to_dev(r), to_dev(F, torch.float32)).cpu().numpy()
    ref = om.apply(r, F.astype(np.float64), om.Params(synth.ETA, A), np.array([0]))
    assert np.abs(U[:, 0, 0] - ref[:, 0, 0]).max() <= 1e-5 * np.abs(ref[:, 0, 0]).max()


@pytest.mark.parametrize("wall,cell", [(True, 0.0), (True, 45.3), (False, 0.0)])
def test_almost_coincident_blobs(wall, cell):
    """Blobs so close that r^-3 overflows: velocities as at the smallest separation whose r^-3 is finite, gradients too
    (they depend on the direction of the separation, however small it is).  The FP64 block and the gradients were
    infinite or NaN between 1e-145 and 1e-103; in FP32 the gradient counts blobs within 2e-13 a as coincident."""
    h = Handle(synth.ETA, A, synth.KT, wall=wall, Lx=cell, Ly=cell)
    r = cloud(40, 950)
    u, F = synth.gaussian(951, (2, 3, 40))
    r[0, :2], r[1:, 1] = 0.0, r[1:, 0]
    calls = [lambda x: h.mobility_apply(x, to_dev(F)), lambda x: h.mobility_adjoint(x, to_dev(u), to_dev(F)),
             lambda x: h.mobility_adjoint(x, to_dev(u), to_dev(F), dtype=F32)]

    def at(gap):
        r[0, 1] = gap
        return [f(to_dev(r)) for f in calls]

    coincident, ref = at(0.0), at(1e-60)
    for gap in (1e-85, 1e-92, 1e-104, 1e-120, 1e-140, 1e-150):
        for i, (g, v, tol) in enumerate(zip(at(gap), (coincident[0], ref[1], coincident[2]), (1e-14, 1e-13, 1e-6))):
            assert float((g - v).norm() / v.norm()) <= tol, (gap, i)
    for gap in (1e-14 * A, 1e-155, 1e-165, 1e-200, 1e-310):
        assert all(torch.isfinite(g).all() for g in at(gap)), gap


# home tiles of one and four warps; the last: one home tile and one item of every step part a launch
@pytest.mark.parametrize("n,kib", [(3000, 1000), (9000, 3000), (700, 200)])
@pytest.mark.parametrize("wall,cell", [(True, 0.0), (True, 45.3), (False, 0.0)])
def test_adjoint_with_little_memory(n, kib, wall, cell):
    """Partials cut into groups of home tiles and, in FP32, of items give the sums of the whole."""
    r = to_dev(cloud(n, 960))
    new = lambda: Handle(synth.ETA, A, synth.KT, wall=wall, Lx=cell, Ly=cell)
    h, g = new(), new()
    h.set_test_memory(kib)
    for k in (1, 6):
        u, F = (to_dev(synth.gaussian(961 + i, (k, 3, n))) for i in range(2))
        for dtype in (F64, F32):
            if dtype == F32 and n == 700:
                h.set_test_memory(300)  # (its records)
            before = h.lib.rpbd_launch_count()
            a = h.mobility_adjoint(r, u, F, dtype=dtype)
            launches = h.lib.rpbd_launch_count() - before
            b = g.mobility_adjoint(r, u, F, dtype=dtype)
            assert launches > 2 * (h.lib.rpbd_launch_count() - before - launches)
            assert float((a - b).norm() / b.norm()) <= 1e-12


def test_adjoint_workspace_is_bounded():
    """The homes' partial rows, one per item, grew with the square of n: 11 GiB at this size."""
    n = 600_000
    args = [to_dev(x) for x in (cloud(n, 970), *synth.gaussian(971, (2, 3, n)))]
    h = Handle(synth.ETA, A, synth.KT)
    out = torch.empty_like(args[0])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    h.mobility_adjoint(*args, out=out, dtype=F32)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 5 << 30  # 4 GiB of partials, an eighth of headroom, records, sums
    assert torch.isfinite(out).all()


@pytest.mark.parametrize("k", [1, 3, 6])
def test_short_memory_is_remembered(k):
    """Where the symmetric FP64 matvec's or the gradients' partials do not fit, the smaller way is taken without asking
    for the memory again: repeated calls can be captured, and one in 256 asks again without harm."""
    n = 3000
    r = to_dev(cloud(n, 980))
    u, F = (to_dev(synth.gaussian(981 + i, (k, 3, n))) for i in range(2))
    h, g = Handle(synth.ETA, A, synth.KT), Handle(synth.ETA, A, synth.KT)
    limits = {1: 4000, 3: 16_000, 6: 32_000}[k], 4000  # KiB: room for the one-direction kernel's partials; a few rows
    calls = [lambda q, out: q.mobility_apply(r, F, out=out), lambda q, out: q.mobility_adjoint(r, u, F, out=out, dtype=F64)]
    for f, like, limit in zip(calls, (F, r), limits):
        h.set_test_memory(limit)
        ref, out = f(g, torch.empty_like(like)), torch.empty_like(like)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            f(h, out)
            assert float((out - ref).norm() / ref.norm()) <= 1e-12
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st):
                f(h, out)
            out.zero_()
            graph.replay()
            assert float((out - ref).norm() / ref.norm()) <= 1e-12
            for _ in range(300):
                out.zero_()
                f(h, out)
            assert float((out - ref).norm() / ref.norm()) <= 1e-12
        st.synchronize()


def test_one_home_list_in_flight():
    """Matvecs without the wall, of other sizes queued behind one another on a stream of their own: the work list was
    rewritten for the next size while the last call read it."""
    h = Handle(synth.ETA, A, synth.KT, wall=False)
    st = torch.cuda.Stream()
    calls = []
    for n in (30_000, 300, 12_001):
        r, F = to_dev(cloud(n, 990)), to_dev(synth.gaussian(991, (3, n)), torch.float32)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            ref = h.mobility_apply(r, F)
            st.synchronize()
            calls.append((r, F, ref))
    with torch.cuda.stream(st):
        outs = [(h.mobility_apply(r, F), ref) for r, F, ref in calls * 3]
        st.synchronize()
    for out, ref in outs:
        assert torch.equal(out, ref)


def test_failed_autotune_changes_nothing():
    """An autotuning run that ends in an error leaves the handle's kernel choice as it was (the one-direction kernel
    stayed chosen, and profiling off)."""
    n = 3000
    r, F = to_dev(cloud(n, 995)), to_dev(synth.gaussian(996, (3, n)), torch.float32)
    h, g = Handle(synth.ETA, A, synth.KT), Handle(synth.ETA, A, synth.KT)
    h.set_test_memory(80)  # KiB: room for the vectors (70), not for records
    h.lib.rpbd_profile_enable(h.h, 1)
    with pytest.raises(RpbdError, match="memory"):
        h.autotune(r)
    h.set_test_memory(0)
    assert torch.equal(h.mobility_apply(r, F), g.mobility_apply(r, F))
    ms, launches, pairs = C.c_double(), C.c_longlong(), C.c_double()
    h.lib.rpbd_profile_read(h.h, 4, 1, C.byref(ms), C.byref(launches), C.byref(pairs), 1)
    assert launches.value == 1


# 4,096 / 4,097: 16 and 64 sources a stage; 4,159 / 4,161: around a whole number of stages of 64
@pytest.mark.parametrize("n", [4096, 4097, 4159, 4161])
@pytest.mark.parametrize("cell", [0.0, 45.3])
def test_many_right_hand_sides_by_stage_length(n, cell):
    r = cloud(n, 1000 + n)
    h = Handle(synth.ETA, A, synth.KT, Lx=cell, Ly=cell)
    rows = np.unique(np.concatenate([[0, 63, 64, 255, 256, n - 66, n - 65, n - 2, n - 1], np.linspace(0, n - 1, 25).astype(int)]))
    for k in (5, 8, 9, 16):
        F = synth.gaussian(1001 + k, (k, 3, n), np.float32)
        U = h.mobility_apply(to_dev(r), to_dev(F, torch.float32)).cpu().numpy()
        ref = om.apply(r, F.astype(np.float64), om.Params(synth.ETA, A, Lx=cell, Ly=cell), rows)
        assert np.linalg.norm(U[:, :, rows] - ref) <= 1e-5 * np.linalg.norm(ref)


def test_fp64_reciprocal_root():
    """Velocities along z of far blobs on the x axis, pulled by one at the origin: 1/r + 2 a^2 / (3 r^3), r from 2.1 a to
    1e100.  The root may be two units of 2^-52 off (one from CUDA's, which may be one off), r^2, the sum and the three
    factors of 1/(8 pi eta) round by half a unit each."""
    n = 2049
    x = np.exp(np.linspace(np.log(2.1 * A), np.log(1e100), n - 1)) * (1 + 0.3 * np.random.default_rng(1010).uniform(size=n - 1))
    r, F = np.zeros((3, n)), np.zeros((3, n))
    r[0, 1:], F[2, 0] = x, 1.0
    eta = 1.0 / (8.0 * np.pi)
    U = Handle(eta, A, synth.KT, wall=False).mobility_apply(to_dev(r), to_dev(F)).cpu().numpy()
    inv8pieta = Fraction(1.0 / (8.0 * np.pi * eta))
    for xi, u in zip(x, U[2, 1:]):
        f = Fraction(float(xi))
        ref = inv8pieta * (1 / f + Fraction(2, 3) * Fraction(float(A)) ** 2 / f ** 3)
        assert abs(Fraction(float(u)) / ref - 1) <= 5 * Fraction(1, 2 ** 52)


def test_square_root_of_one_number():
    """M^(1/2) W of a lone unbounded blob, over two octaves of its mobility: sqrt(1 / (6 pi eta a)) W.  Nodes and weights
    are good to 5e-15, 64 rounded terms add 7e-15, the pivots' reciprocals and the norms a few units of 2^-52."""
    W = to_dev(synth.gaussian(1011, (3, 1)))
    r = torch.zeros_like(W)
    for eta in np.geomspace(1e-3, 4e-3, 65):
        out, _ = Handle(eta, A, synth.KT, wall=False).lanczos_sqrt_apply(r, W, tol=1e-14, use_precond=False)
        ref = np.sqrt(1.0 / (6.0 * np.pi * eta * A)) * W
        assert float((out - ref).norm() / ref.norm()) <= 2e-14


@pytest.mark.parametrize("wall", [True, False])
def test_blobs_beyond_the_square_root_of_the_range(wall):
    """Blobs so far apart that r^2 overflows do not feel one another (1/r was NaN there, in FP64)."""
    h = Handle(synth.ETA, A, synth.KT, wall=wall)
    r, F = cloud(80, 1020), synth.gaussian(1021, (3, 80))
    near = [h.mobility_apply(to_dev(r[:, s]), to_dev(F[:, s])) for s in (slice(0, 40), slice(40, 80))]
    r[0, 40:] = 1e160  # (all of them on one line along y)
    far = h.mobility_apply(to_dev(r), to_dev(F))
    assert torch.allclose(far[:, :40], near[0], rtol=1e-13, atol=1e-13 * float(near[0].abs().max()))
    assert torch.isfinite(far).all()
