"""Infinite and very large values: the kernels that split their operands give what plain fp32 arithmetic gives."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def run(api, Q, K, V, scale, variant=0, **kw):
    O = torch.full_like(Q, 7.0)
    lse = torch.full(Q.shape[:3], 7.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.flat_attn_fwd_ex(Q, K, V, O, scale, status=status, variant=variant, lse=lse, **kw)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return O.float(), lse


def check(api, Q, K, V, scale, variant, rounding, **kw):
    """AUTO (which must run `variant`) against the FFMA kernel: the same infinities and NaN, finite values to `rounding` of the
    largest value a feature has (each is off the exact one by its format's rounding, and by sums in another order)."""
    O, lse = run(api, Q, K, V, scale, **kw)
    assert api.flat_attn_last_variant() == variant
    F, flse = run(api, Q, K, V, scale, variant=api.FLAT_VARIANT_SIMT, **kw)
    for got, want, size in ((O, F, V.float().nan_to_num(0.0, 0.0, 0.0).abs().amax(2, keepdim=True)), (lse, flse, None)):
        same = (got == want) | (got.isnan() & want.isnan())
        ok = got.isfinite() & want.isfinite()
        bound = rounding * size if size is not None else 4e-5 * (1 + want.abs())
        near = ok & ((got - want).abs() <= bound)
        assert bool((same | near).all())
    return O


FORMATS = [(16, torch.bfloat16), (32, torch.bfloat16), (32, torch.float32), (128, torch.float32)]


def variant_of(api, dtype):
    return api.FLAT_VARIANT_SMALL if dtype == torch.bfloat16 else api.FLAT_VARIANT_TF32


def rounding_of(dtype):                                  # of one bf16 number (2^-8), or of fp32 sums of a few hundred terms
    return 2.0 ** -7 if dtype == torch.bfloat16 else 2.0 ** -16


@pytest.mark.parametrize("d,dtype", FORMATS)
@pytest.mark.parametrize("options", [{}, {"causal": True}, {"valid": True}], ids=str)
def test_infinite_values(d, dtype, options):
    from paper_2107_06419_b200 import api
    torch.manual_seed(d)
    B, H, Nq, Nk = 2, 3, 150, 333
    Q, K, V = (torch.randn(B, H, n, d, device="cuda").to(dtype) for n in (Nq, Nk, Nk))
    V[0, 0, 5, 1] = float("inf")
    V[0, 0, 6, 2] = -float("inf")
    V[0, 1, 7, 3], V[0, 1, 140, 3] = float("inf"), -float("inf")   # both signs in one feature: NaN where a row sees both
    V[1, 0, 9, 0] = float("nan")
    K[1, 1, 20, 4] = float("inf")                        # an infinite logit of either sign
    Q[1, 2, 30, 5] = -float("inf")
    kw = {"causal": True} if "causal" in options else {}
    if "valid" in options:
        kw["k_valid_len"] = torch.tensor([333, 50], dtype=torch.int32, device="cuda")
    O = check(api, Q, K, V, d ** -0.5, variant_of(api, dtype), rounding_of(dtype), **kw)
    assert bool((O[0, 0, :, 1] == float("inf")).all()) and bool((O[0, 0, :, 2] == -float("inf")).all())
    rest = [c for c in range(d) if c not in (1, 2)]
    assert bool(O[0, 0][:, rest].isfinite().all())


@pytest.mark.parametrize("d,dtype", FORMATS)
def test_large_values_behind_growing_logits(d, dtype):
    """A few keys whose logits lie 36 (base 2) above the first ones', with values about 2^100: weight times value passes the largest
    number, while the sum of the weights stays below the bound that has a step redone."""
    from paper_2107_06419_b200 import api
    torch.manual_seed(d + 1)
    Q = torch.ones(1, 2, 140, d, device="cuda", dtype=dtype)
    K = torch.zeros(1, 2, 500, d, device="cuda", dtype=dtype)
    K[:, :, 200:203] = 25.0 / d
    V = torch.randn(1, 2, 500, d, device="cuda").to(dtype) * 2.0 ** 100
    O = check(api, Q, K, V, 1.0, variant_of(api, dtype), rounding_of(dtype))
    assert bool(O.isfinite().all())
    f64 = lambda t: t.double().cpu().numpy()
    x = f64(Q)[0] @ f64(K)[0].transpose(0, 2, 1)
    p = np.exp(x - x.max(-1, keepdims=True))
    ref = (p / p.sum(-1, keepdims=True)) @ f64(V)[0]
    assert np.max(np.abs(f64(O)[0] - ref)) <= rounding_of(dtype) * np.abs(f64(V)).max()


@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("key", [5, 70, 100])            # in an even and in an odd key step
def test_nan_inputs_leave_no_row_unwritten(d, key):
    """A NaN logit makes its row NaN, as on the FFMA kernel; the row must not keep what the output held before."""
    from paper_2107_06419_b200 import api
    torch.manual_seed(key)
    Q, K, V = (torch.randn(1, 2, n, d, device="cuda") for n in (140, 200, 200))
    K[0, 0, key, 3] = float("nan")
    Q[0, 1, 20, 1] = float("nan")
    O, lse = run(api, Q, K, V, d ** -0.5)
    F, flse = run(api, Q, K, V, d ** -0.5, variant=api.FLAT_VARIANT_SIMT)
    assert bool(O[0, 0].isnan().all()) and bool(O[0, 1, 20].isnan().all())
    assert torch.equal(O.isnan(), F.isnan()) and torch.equal(lse.isinf(), flse.isinf()) and bool((lse[0, 1, :20] != 7.0).all())


@pytest.mark.parametrize("d,dtype", FORMATS)
@pytest.mark.parametrize("rows", [1, 7, 8, 9, 31])
def test_some_rows_of_a_warp(d, dtype, rows):
    """As many rows of a warp come out NaN (a NaN in their query) as the second pass takes at a time, less and more; an infinite value
    under the causal mask is seen by the later rows only."""
    from paper_2107_06419_b200 import api
    torch.manual_seed(rows)
    Q, K, V = (torch.randn(1, 2, 160, d, device="cuda").to(dtype) for _ in range(3))
    Q[0, 0, 33:33 + rows, 2] = float("nan")
    V[0, 1, 160 - rows, 3] = float("inf")
    O, lse = run(api, Q, K, V, d ** -0.5, causal=True)
    assert api.flat_attn_last_variant() == variant_of(api, dtype)
    bad = O[0, 0].isnan()
    assert bool(bad[33:33 + rows].all()) and int(bad.sum()) == rows * d
    assert int((O[0, 1] == float("inf")).sum()) == rows and bool((O[0, 1, 160 - rows:, 3] == float("inf")).all())
    ref = torch.softmax((Q.double() @ K.double().transpose(2, 3) * d ** -0.5).masked_fill(
        torch.ones(160, 160, device="cuda", dtype=torch.bool).triu(1), -float("inf")), -1) @ V.double().nan_to_num(0.0, 0.0, 0.0)
    ok = O.isfinite()
    assert int(ok.sum()) == O.numel() - rows * d - rows
    assert float((O.double() - ref)[ok].abs().max()) <= rounding_of(dtype) * float(V.float().nan_to_num(0.0, 0.0, 0.0).abs().max())
