"""The level scans at the sizes where their tiles, chunks and packed trees can
go wrong: refinement flags equal the oracle's byte for byte (tiles that
just fit, one cell more, one cell, more planes than a chunk, decisions at the rounding
limit, huge, tiny and non-finite values), conservation sums equal the
allocation-free ones bit for bit (cell volumes that are and are not powers of
two, FP32 subnormals, blocks with a remainder)."""
import numpy as np
import pytest
import torch

from gpu_util import random_state, to_patch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    from paper_1112_1710_gb300 import _build, capi as C
    _build.build()
    C.load()
    return C


SIZES = [(5, 9, 18), (8, 49, 1), (16, 17, 33), (30, 14, 16), (31, 15, 17), (70, 31, 20), (1, 1, 1)]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("theta", [0.0, 0.11, 0.3, 1.5])
@pytest.mark.parametrize("scale", [1.0, 1e-34, 1e33, "special"])
def test_flags_equal_oracle(capi, orc, dtype, theta, scale):
    from paper_1112_1710_gb300 import regrid
    ctx = capi.mhd_ctx_create()
    try:
        pats, want = [], []
        for m, n in enumerate(SIZES):
            st = random_state(n, 2, seed=90 + m)
            if scale == "special":
                rng = np.random.default_rng(m)
                # ties: neighbouring cells equal or off by one unit, and values no
                # bound holds for
                st[0] = np.where(rng.random(st.shape[1:]) < 0.5, 1.0, 1.0 + 2.0 ** -23)
                for v in (0.0, -1.0, np.inf, np.nan, 1e-42, 3e38):
                    st[rng.integers(0, 5, 9), rng.integers(0, st.shape[1], 9), rng.integers(0, st.shape[2], 9),
                       rng.integers(0, st.shape[3], 9)] = v
            else:
                st[1:5] *= scale
                st[0] *= scale
                st[5:8] *= np.sqrt(scale)
            p = to_patch(st, n, 2, (0.1, 0.1, 0.1), dtype=dtype)
            pats.append(p)
            seen = np.ascontiguousarray(p.state.cpu().numpy().astype(np.float64))
            with np.errstate(all="ignore"):
                want.append(orc.flag(orc.patch(seen, n, 2, (0.1, 0.1, 0.1)), orc.params(), theta))
        got = regrid.flag(ctx, pats, theta)
        torch.cuda.synchronize()
        for n, f, w in zip(SIZES, got, want):
            assert np.array_equal(f.cpu().numpy(), w), n
    finally:
        capi.mhd_ctx_destroy(ctx)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("dx", [(0.25, 0.5, 0.125), (0.1, 0.3, 0.07), (2.0 ** -20, 2.0 ** -300, 2.0 ** -200)])
def test_sums_equal_static(capi, dtype, dx):
    ctx = capi.mhd_ctx_create()
    try:
        pats = []
        for m, n in enumerate(SIZES):
            st = random_state(n, 2, seed=40 + m)
            st[1] *= 1e-40      # FP32 subnormals and zeros
            st[2] *= -1.0
            st[3, ::2] = 0.0
            pats.append(to_patch(st, n, 2, dx, dtype=dtype))
        descs = [p.desc() for p in pats]
        a = torch.zeros(8, dtype=torch.float64, device="cuda")
        b = torch.zeros(8, dtype=torch.float64, device="cuda")
        capi.mhd_conservation_sums(ctx, descs, a.data_ptr())
        capi.mhd_conservation_sums_static(descs, b.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))
        assert bool((a != 0).any())
    finally:
        capi.mhd_ctx_destroy(ctx)
