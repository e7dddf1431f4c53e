"""How an untuned FP32 advance is run: the fused pass where the dt is given, and the
upwinded edge EMFs from a kernel of their own from a size on, against the
other form of each."""
import numpy as np
import pytest
import torch

from gpu_util import random_state, rel_linf, to_patch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    from paper_1112_1710_gb300 import capi as c
    return c


def _advance(capi, st, n, g, k, copies=1, cfl=False, **prm):
    """The first of `copies` equal FP32 patches after one advance."""
    dx = (0.05, 0.07, 0.06)
    ctx = capi.mhd_ctx_create(**prm)
    try:
        p = [to_patch(st.copy(), n, g, dx, dtype="f32", pid=i) for i in range(copies)]
        d = torch.full((1,), 1.2e-3, dtype=torch.float64, device="cuda")
        if cfl:
            capi.mhd_patch_step_cfl(ctx, [q.desc() for q in p], d.data_ptr())
        else:
            capi.mhd_patch_advance(ctx, [q.desc() for q in p], d.data_ptr(), grow=[k] * copies)
        assert capi.mhd_get_device_status(ctx) == 0
        return p[0].state.cpu().numpy()
    finally:
        capi.mhd_ctx_destroy(ctx)


# FP32 bound: one step is a few hundred operations of rounding 6e-8 on values of
# order one, most of them averaged out: 1e-5, as for the other FP32 comparisons
TOL32 = 1e-5


@pytest.mark.parametrize("emf,lim", [(0, 0), (1, 2), (0, 1)])
@pytest.mark.parametrize("n,k,chunk", [((14, 30, 9), 0, 0), ((15, 13, 11), 2, 0), ((31, 33, 6), 1, 3), ((5, 16, 1), 0, 1)])
def test_fused_pass_fp32_close_to_staged(capi, n, k, chunk, emf, lim):
    """Tiles of exactly 16 cells, one more and one less, partial chunks, one
    plane, and columns shorter than the ring."""
    st = random_state(n, 4, seed=91 + k)
    a = _advance(capi, st, n, 4, k, emf=emf, limiter=lim, advance_kernel=1)
    for shape in (1, 2, 3, 4):
        b = _advance(capi, st, n, 4, k, emf=emf, limiter=lim, advance_kernel=4, fused_chunk=chunk, kernel_shape=shape)
        assert rel_linf(b, a.astype(np.float64), n, 4).max() <= TOL32, shape


@pytest.mark.parametrize("n", [(40, 40, 40), (80, 77, 75), (300, 300, 1)])
def test_untuned_fp32_route(capi, n):
    """An untuned context gives the bits of the form its call selects: with a given
    dt the fused pass, with the CFL dt or a grown update box the staged kernels."""
    st = random_state(n, 4, seed=17)
    for cfl, k, pf in ((True, 0, False), (False, 0, True), (False, 1, False)):
        a = _advance(capi, st, n, 4, k, cfl=cfl, emf=0)
        b = _advance(capi, st, n, 4, k, cfl=cfl, emf=0, advance_kernel=4 if pf else 1)
        assert np.array_equal(a, b), (cfl, k)


@pytest.mark.parametrize("kernel", [1, 4])
def test_upwinded_emf_kernel_equals_inline(capi, kernel):
    """One small patch (edge EMFs inside the update) and the same patch in a
    batch of over a block per SM (edge EMFs by their own kernel): the same bits."""
    n = (17, 12, 14)
    st = random_state(n, 4, seed=29)
    a = _advance(capi, st, n, 4, 1, emf=0, advance_kernel=kernel)
    b = _advance(capi, st, n, 4, 1, copies=40, emf=0, advance_kernel=kernel)
    assert np.array_equal(a, b)
