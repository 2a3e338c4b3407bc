"""The host call works in slices of batches or heads: a bias and a pruning map that differ from one to the next go with them."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["bias", "bias f32", "map"])
@pytest.mark.parametrize("B,H", [(3, 2), (1, 5)])
def test_bias_and_map_per_slice(B, H, what):
    from paper_2107_06419_b200 import api
    torch.manual_seed(B)
    Nq, Nk, d = 200, 328, 64
    Q, K, V = (torch.randn(B, H, n, d).to(torch.bfloat16).pin_memory() for n in (Nq, Nk, Nk))
    O = torch.zeros_like(Q).pin_memory()
    ws = torch.empty(api.flat_attn_host_workspace_bytes(B, H, Nq, Nk, d), dtype=torch.uint8, device="cuda")
    p = api._params(Q, K, V, O, 0.125, None, None, 0, host=True)
    kw = {}
    if what == "map":
        kw["block_mask"] = (torch.rand(B, H, 2, 3, device="cuda") < 0.6).to(torch.uint8)
        p.block_mask, p.block_mask_stride_h, p.block_mask_stride_b = kw["block_mask"].data_ptr(), 6, 6 * H
    else:
        dtype = torch.float32 if "f32" in what else torch.bfloat16
        kw["bias"] = torch.randn(B, H, Nq, Nk, device="cuda").to(dtype)
        p.bias, p.bias_dtype = kw["bias"].data_ptr(), api.FLAT_DTYPE_F32 if dtype == torch.float32 else api.FLAT_DTYPE_BF16
        p.bias_stride_h, p.bias_stride_b = Nq * Nk, H * Nq * Nk
    api._check(api._lib.flat_attn_fwd_host(ctypes.byref(p), ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    want = torch.empty_like(Q, device="cuda")
    api.flat_attn_fwd_ex(Q.cuda(), K.cuda(), V.cuda(), want, 0.125, **kw)
    torch.cuda.synchronize()
    # (a slice may take another dispatch than the whole: one rounding of a bf16 result)
    assert float((O.cuda().float() - want.float()).abs().max()) <= 2.0 ** -7 * float(V.float().abs().max())
