"""Key counts beyond what a kernel's index arithmetic holds are refused when it is asked for by name (AUTO then takes another)."""
import ctypes

import pytest


@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("Nk", [2 ** 30 + 1, 2 ** 31 - 1])
def test_small_heads(d, Nk):
    from paper_2107_06419_b200 import api
    p = api.flat_attn_params_t()
    p.Q, p.K, p.V, p.O = 0x10000, 0x20000, 0x30000, 0x40000     # never dereferenced: refused before a launch
    p.B, p.H, p.Nq, p.Nk, p.d, p.scale, p.dtype, p.variant = 1, 1, 1, Nk, d, 1.0, api.FLAT_DTYPE_BF16, api.FLAT_VARIANT_SMALL
    assert api._lib.flat_attn_fwd_ex(ctypes.byref(p), None) == 3
