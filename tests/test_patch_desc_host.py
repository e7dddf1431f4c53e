"""Patch.desc() packs the descriptor's fields as ctypes assignments would: any
integer type, and integers beyond 32 bits (a request counter or a hash as patch
id) modulo 2^32 -- no GPU."""
import ctypes

import numpy as np
import pytest

from paper_1112_1710_gb300 import capi
from paper_1112_1710_gb300.patch import Patch


class _State:
    """What desc() asks of a contiguous CUDA state tensor."""
    is_cuda, dtype = True, None

    def is_contiguous(self):
        return True

    def stride(self):
        return (9 * 7 * 16, 7 * 16, 16, 1)

    def data_ptr(self):
        return 0x7f0000001000

    def element_size(self):
        return 4


@pytest.mark.parametrize("level,pid,lo", [(0, 0, (0, 0, 0)), (3, 2 ** 31 - 1, (-4, 7, 10 ** 6)), (1, 2 ** 31, (0, 0, 0)),
                                          (1, -2 ** 31 - 1, (0, 0, 0)), (0, 2 ** 40 + 17, (2 ** 31, 0, -2 ** 33)),
                                          (np.int64(2), np.int64(2 ** 35 + 1), (np.int32(1), np.int64(2), 3)), (True, 5, (0, 1, 2))])
def test_desc_fields(level, pid, lo):
    n, g, dx = (11, 3, 4), 2, (0.5, 0.25, 0.125)
    p = Patch(_State(), lo, n, g, dx, level, pid)
    d = capi.mhd_patch_desc()
    d.level, d.nghost, d.dtype, d.patch_id = int(level), g, capi.MHD_F32, int(pid)
    d.interior.lo[:] = [int(v) for v in lo]
    d.interior.hi[:] = [int(lo[a]) + n[a] - 1 for a in range(3)]
    for q in range(5):
        d.U[q] = 0x7f0000001000 + q * 9 * 7 * 16 * 4
    for a in range(3):
        d.B[a] = 0x7f0000001000 + (5 + a) * 9 * 7 * 16 * 4
    d.stride[:] = (1, 16, 7 * 16)
    d.dx[:] = dx
    assert bytes(p.desc()) == bytes(d)
    assert ctypes.sizeof(d) == len(bytes(d))


@pytest.mark.parametrize("level,pid", [(1.0, 0), (0, 1.5), (0, None), ("1", 0)])
def test_desc_refuses_what_is_no_integer(level, pid):
    with pytest.raises(TypeError):
        Patch(_State(), (0, 0, 0), (4, 4, 4), 2, (1.0,) * 3, level, pid).desc()
