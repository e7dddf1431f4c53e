"""What mhd_params.advance_kernel may change: nothing in the FP64 parity build;
rounding in the contracted FP64 build and in FP32."""
import numpy as np
import pytest

from gpu_util import rel_linf
from test_gpu_fp32_forms import _moving, capi  # noqa: F401 (fixture)
import test_gpu_fp32_forms as forms

pytestmark = pytest.mark.gpu


def _advance(capi, st, n, k, dt, dtype, **prm):  # noqa: F811
    import torch
    from gpu_util import to_patch
    ctx = capi.mhd_ctx_create(**prm)
    try:
        p = to_patch(st.copy(), n, 4, forms.DX, dtype=dtype)
        d = torch.full((1,), dt, dtype=torch.float64, device="cuda")
        capi.mhd_patch_advance(ctx, [p.desc()], d.data_ptr(), grow=[k])
        return p.state.cpu().numpy()
    finally:
        capi.mhd_ctx_destroy(ctx)


# the bounds: a step is a few hundred operations of rounding 1.1e-16 (FP64) or 6e-8
# (FP32) on values of order one, most of them averaged out
@pytest.mark.parametrize("dtype,contract,tol", [("f64", 0, 0.0), ("f64", 1, 2e-14), ("f32", 0, 1e-5)])
@pytest.mark.parametrize("emf,lim", [(0, 0), (1, 1), (0, 2)])
@pytest.mark.parametrize("mach,floors", [(0.3, {}), (3.0, dict(p_floor=0.1, rho_floor=0.6))])
def test_kernels_agree(capi, dtype, contract, tol, emf, lim, mach, floors):  # noqa: F811
    n, k = (31, 33, 6), 1
    st = _moving(n, 4, 41, mach)
    prm = dict(emf=emf, limiter=lim, fp64_contract=contract, **floors)
    a = _advance(capi, st, n, k, 2e-3 / mach, dtype, advance_kernel=1, **prm)
    for kernel in (2, 3, 4):
        b = _advance(capi, st, n, k, 2e-3 / mach, dtype, advance_kernel=kernel, **prm)
        if tol == 0.0 or (dtype == "f32" and kernel == 4):
            assert np.array_equal(a, b), kernel
        else:
            assert rel_linf(b, a.astype(np.float64), n, 4).max() <= tol, kernel
