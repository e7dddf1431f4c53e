"""Refinement flags of states in units that make the values small (densities
and momenta whose squares leave FP32's range, as in CGS): byte for byte those of
the oracle's FP64 decision."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import random_state, to_patch

pytestmark = pytest.mark.gpu

DX = (0.1, 0.1, 0.1)
SIZES = [(9, 17, 33), (31, 15, 17)]


@pytest.fixture(scope="module")
def capi():
    from paper_1112_1710_gb300 import _build, capi as C
    _build.build()
    C.load()
    return C


def _compare(capi, orc, states, theta, dtype):
    from paper_1112_1710_gb300 import regrid
    ctx = capi.mhd_ctx_create()
    try:
        pats = [to_patch(st, n, 2, DX, dtype=dtype) for st, n in zip(states, SIZES)]
        got = regrid.flag(ctx, pats, theta)
        torch.cuda.synchronize()
        for p, n, f in zip(pats, SIZES, got):
            seen = np.ascontiguousarray(p.state.cpu().numpy().astype(np.float64))
            want = orc.flag(orc.patch(seen, n, 2, DX), orc.params(), theta)
            assert np.array_equal(f.cpu().numpy(), want), (n, int((f.cpu().numpy() != want).sum()))
    finally:
        capi.mhd_ctx_destroy(ctx)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("scale", [10.0 ** -k for k in range(19, 31)])
def test_flags_of_scaled_states(capi, orc, dtype, field, scale):
    """Cells of order one times `scale` (momenta and density alike, so that the
    velocities stay of order one), with and without a field."""
    states = []
    for m, n in enumerate(SIZES):
        st = random_state(n, 2, seed=300 + m)
        st[4] -= 2.4  # thermal and kinetic energy alike
        st[0:5] *= scale
        st[5:8] *= np.sqrt(scale) if field else 0.0
        states.append(st)
    _compare(capi, orc, states, 0.15, dtype)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("rho,v", [(1e-29, 1e6), (1e-28, 1e5), (1e-26, 1e5), (1e-24, 1e4), (1e-24, 1e6)])
@pytest.mark.parametrize("theta", [0.02, 0.11])
def test_flags_of_uniform_pressure_in_cgs_units(capi, orc, dtype, rho, v, theta):
    """Uniform density and pressure, velocities between 0.3 v and 2 v: what the
    kinetic energy loses the pressure shows."""
    states = []
    for m, n in enumerate(SIZES):
        rng = np.random.default_rng(70 + m)
        st = synth.empty_patch(n, 2, align=8)
        u = rng.uniform(0.3, 2.0, (3,) + st.shape[1:]) * v
        st[0] = rho
        st[1:4] = rho * u
        st[4] = 0.1 * rho * v * v / (2.0 / 3.0) + 0.5 * rho * (u ** 2).sum(0)
        states.append(st)
    _compare(capi, orc, states, theta, dtype)
