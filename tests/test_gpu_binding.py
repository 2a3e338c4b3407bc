"""The native way into the library and the long one (arguments that are not plain) give the same results and the same errors."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("options", [{}, {"valid": True}, {"causal": True, "lse": True}, {"bias": (1, 2)}, {"bias": (2, 1)}, {"map": True}],
                         ids=str)
def test_forward_both_ways(dtype, options):
    from paper_2107_06419_b200 import api
    if dtype == torch.float32 and "map" in options:
        pytest.skip("the pruning map is bf16 only")
    torch.manual_seed(3)
    B, H, Nq, Nk, d = 2, 2, 200, 300, 64
    Q, K, V = (torch.randn(B, H, n, d, device="cuda").to(dtype) for n in (Nq, Nk, Nk))
    kw = {"causal": bool(options.get("causal"))}
    if options.get("valid"):
        kw["k_valid_len"] = torch.tensor([300, 77], dtype=torch.int32, device="cuda")
    if options.get("bias"):
        kw["bias"] = torch.randn(options["bias"] + (Nq, Nk), device="cuda").to(torch.bfloat16)
    if options.get("map"):
        kw["block_mask"] = (torch.rand(1, H, 2, 3, device="cuda") < 0.7).to(torch.uint8)
    out = []
    for scale in (0.125, np.float64(0.125)):             # (a numpy scalar is not plain: the long way)
        assert (api._binding.fwd(Q, K, V, torch.empty_like(Q), scale, None) >= 0) == (type(scale) is float and dtype == torch.bfloat16)
        O = torch.full_like(Q, float("nan"))
        lse = torch.full((B, H, Nq), float("nan"), device="cuda") if options.get("lse") else None
        api.flat_attn_fwd_ex(Q, K, V, O, scale, lse=lse, stream=torch.cuda.current_stream(), **kw)
        torch.cuda.synchronize()
        out.append((O, lse if lse is not None else O))
    assert all(torch.equal(a, b) for a, b in zip(*out)) and torch.isfinite(out[0][0]).all()


def test_errors_are_those_of_the_long_way():
    from paper_2107_06419_b200 import api
    q = torch.zeros(1, 1, 128, 64, dtype=torch.bfloat16, device="cuda")
    o = torch.empty_like(q)
    for bad, error in (((q, q[:, :, :, :32], q, o), ValueError), ((q, q, q.float(), o), TypeError), ((q.cpu(), q, q, o), ValueError),
                       ((q, q, q.transpose(2, 3), o), ValueError), ((q.half(), q.half(), q.half(), o.half()), TypeError)):
        with pytest.raises(error):
            api.flat_attn_fwd(*bad, 0.125)
    with pytest.raises(api.FlatAttnError) as e:
        api.flat_attn_fwd(q, q, q, o, float("nan"))
    assert e.value.code == 2
    with pytest.raises(ValueError):
        api.flat_attn_fwd_ex(q, q, q, o, 0.125, k_valid_len=torch.zeros(2, dtype=torch.int32, device="cuda"))
