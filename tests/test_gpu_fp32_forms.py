"""FP32: the staged kernels and the fused pass give the same bits, so that what
an untuned context picks for a call (by its captures, grown boxes and dt) never
shows in the state: patches of one level advanced in different calls agree on
their shared faces, and a patch gives the same bits alone and in any batch."""
import numpy as np
import pytest
import torch

import synth
import synth.amr as SA
import synth.turb as ST
from gpu_util import random_state, to_patch

pytestmark = pytest.mark.gpu
DX = (0.05, 0.07, 0.06)


@pytest.fixture(scope="module")
def capi():
    from paper_1112_1710_gb300 import _build, capi as C
    _build.build()
    C.load()
    return C


def _moving(n, g, seed, mach):
    """random_state with velocities up to `mach` along each axis (slow: all
    HLLD states inside the fan; fast: supersonic and single-star faces) and in
    a tenth of the cells 1% of the pressure (positivity rules)."""
    st = random_state(n, g, seed=seed)
    rng = np.random.default_rng(seed)
    p = rng.uniform(0.5, 1.5, st.shape[1:]) * np.where(rng.random(st.shape[1:]) < 0.1, 0.01, 1.0)
    st[1:4] *= 2.0 * mach * st[0]
    st[4] = 1.5 * p + 0.5 * (st[1:4] ** 2).sum(0) / st[0] + 0.5 * 3 * 0.7 ** 2
    return st


def _advance(capi, st, n, g, k, dt, **prm):
    ctx = capi.mhd_ctx_create(**prm)
    try:
        p = to_patch(st.copy(), n, g, DX, dtype="f32")
        d = torch.full((1,), dt, dtype=torch.float64, device="cuda")
        capi.mhd_patch_advance(ctx, [p.desc()], d.data_ptr(), grow=[k])
        return p.state.cpu().numpy()
    finally:
        capi.mhd_ctx_destroy(ctx)


@pytest.mark.parametrize("emf,lim", [(0, 0), (1, 0), (0, 1), (1, 2)])
@pytest.mark.parametrize("mach,floors", [(0.3, {}), (3.0, {}), (3.0, dict(p_floor=0.1, rho_floor=0.6))])
@pytest.mark.parametrize("n,k,chunk", [((14, 30, 9), 0, 0), ((15, 13, 11), 2, 0), ((31, 33, 6), 1, 3), ((5, 16, 1), 0, 1),
                                       ((48, 40, 37), 0, 0)])
def test_fused_pass_fp32_equals_staged_bitexact(capi, n, k, chunk, emf, lim, mach, floors):
    """Every compiled shape, over tiles of exactly 16 cells, one more and one
    less, partial chunks, one plane and columns shorter than the ring."""
    st = _moving(n, 4, 40 + k, mach)
    prm = dict(emf=emf, limiter=lim, **floors)
    a = _advance(capi, st, n, 4, k, 2e-3 / mach, advance_kernel=1, **prm)
    for shape in (1, 2, 3, 4):
        b = _advance(capi, st, n, 4, k, 2e-3 / mach, advance_kernel=4, fused_chunk=chunk, kernel_shape=shape, **prm)
        assert np.array_equal(a.view(np.int32), b.view(np.int32)), shape


def test_mixed_call_equals_each_patch_alone(capi):
    """One call with a captured patch, a grown one and plain ones against a
    call for each, untuned: states and captured fluxes."""
    sizes, grow = [(17, 12, 14), (20, 16, 9), (33, 8, 21), (6, 6, 6)], [0, 1, 0, 0]
    states = [_moving(n, 4, 60 + i, 0.7) for i, n in enumerate(sizes)]
    d = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
    out = []
    for together in (True, False):
        ctx = capi.mhd_ctx_create()
        ps = [to_patch(s.copy(), n, 4, DX, dtype="f32", lo=(40 * i, 0, 0), pid=i) for i, (s, n) in enumerate(zip(states, sizes))]
        nx, ny, nz = sizes[0]
        reg = torch.zeros((8, nz, ny, 1), dtype=torch.float64, device="cuda")
        c = capi.mhd_capture()
        c.patch, c.kind, c.axis, c.mode = 0, capi.MHD_CAP_FACE, 0, 0
        c.box = capi.box((0, 0, 0), (0, ny - 1, nz - 1))
        c.dst = reg.data_ptr()
        try:
            if together:
                capi.mhd_patch_advance(ctx, [p.desc() for p in ps], d.data_ptr(), grow=grow, caps=[c])
            else:
                for i, p in enumerate(ps):
                    capi.mhd_patch_advance(ctx, [p.desc()], d.data_ptr(), grow=[grow[i]], caps=[c] if i == 0 else None)
            torch.cuda.synchronize()
            out.append([p.state.cpu().numpy() for p in ps] + [reg.cpu().numpy()])
        finally:
            capi.mhd_ctx_destroy(ctx)
    assert np.any(out[0][-1] != 0)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("kind", ["block", "turbulent"])
def test_hierarchy_fp32_per_patch_equals_batched(capi, kind):
    """Two coarse steps of an FP32 hierarchy with one call per patch (some of a
    level captured, some not) and with one call per level, untuned."""
    from paper_1112_1710_gb300.amr import Hierarchy
    n0, g = 16, 4
    if kind == "block":  # the fine level's central patch has fine neighbours only
        cut = [(4, 11), (12, 19), (20, 27)]
        H = [[((0, 0, 0), (n0 - 1,) * 3)],
             [((x[0], y[0], z[0]), (x[1], y[1], z[1])) for z in cut for y in cut for x in cut]]
        st = [[SA.blast_patch(lo, hi, l, n0, g)[0] for (lo, hi) in bl] for l, bl in enumerate(H)]
    else:
        H, v, _ = ST.deep_hierarchy(n0=n0, levels=3, m=32, size_min=4, size_max=8)
        st = [[ST.turb_patch(lo, hi, l, n0, g, v)[0] for (lo, hi) in bl] for l, bl in enumerate(H)]
    ctx = capi.mhd_ctx_create()
    hs = []
    try:
        for batched in (True, False):
            h = Hierarchy(H, n0, st, (1.0 / n0,) * 3, g=g, dtype="f32", ctx=ctx)
            h.batched = batched
            h.initialise()
            for _ in range(2):
                h.coarse_step()
            hs.append(h)
        torch.cuda.synchronize()
        for la, lb in zip(hs[0].levels, hs[1].levels):
            for pa, pb in zip(la, lb):
                assert np.array_equal(pa.state.cpu().numpy(), pb.state.cpu().numpy())
    finally:
        for h in hs:
            h.close()
        capi.mhd_ctx_destroy(ctx)


@pytest.mark.parametrize("sizes,fused", [([(220, 220, 1)], False), ([(230, 230, 1)], True), ([(59, 60, 60)], False),
                                         ([(60, 60, 60)], True), ([(8, 8, 8)] * 151, False), ([(8, 8, 8)] * 152, True)])
def test_untuned_route_by_size(capi, sizes, fused):
    """Kernel launches of an untuned call on both sides of 2^18 grown cells
    (arithmetic-mean EMF: five staged, three with the fused pass), and the bits of
    the staged kernels either way."""
    out = []
    for kernel in (0, 1):
        ctx = capi.mhd_ctx_create(emf=1, advance_kernel=kernel)
        ps = [to_patch(_moving(n, 2, 5, 0.5), n, 2, DX, dtype="f32", pid=i) for i, n in enumerate(sizes)]
        d = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
        try:
            before = capi.mhd_launch_count(ctx)
            capi.mhd_patch_advance(ctx, [p.desc() for p in ps], d.data_ptr())
            assert capi.mhd_launch_count(ctx) - before == (3 if fused and kernel == 0 else 5)
            out.append([p.state.cpu().numpy() for p in ps])
        finally:
            capi.mhd_ctx_destroy(ctx)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [(100, 40, 40), (31, 29, 102)])
def test_autotune_reports_the_planes_it_timed(capi, n):
    """The reported chunk is one that was timed: a listed length, or the one the
    fused pass picks by itself (a listed length or the whole column)."""
    ctx = capi.mhd_ctx_create(emf=1)
    try:
        p = to_patch(_moving(n, 2, 3, 0.3), n, 2, DX, dtype="f32")
        d = torch.full((1,), 1e-3, dtype=torch.float64, device="cuda")
        for _ in range(3):
            choice, chunk, _ms = capi.mhd_autotune_advance(ctx, [p.desc()], d.data_ptr(), reps=1)
            top = n[2] + 2
            lengths = (2, 3, 4, 5, 6, 8, 10, 12, 14, 16, 20, 24, 28, 33, 40, 48, 66, 88, 130)
            if choice <= -3:
                assert chunk in {min(c, top) for c in lengths}, (choice, chunk)
    finally:
        capi.mhd_ctx_destroy(ctx)
