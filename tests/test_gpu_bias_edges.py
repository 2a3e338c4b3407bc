"""The additive bias where its kernels change: the staged tiles of the d = 64 kernel (several items per CTA, ring of three tiles,
masks, rows and whole tiles of -inf, negative scale, lse) and rows that begin at any alignment."""
import numpy as np
import pytest
import torch

import oracle
from paper_2107_06419_b200 import inputs
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, Nq, Nk, d, bias heads/batches, dtype, valid lengths, causal, scale
    (1, 1, 1, 8, 64, (1, 1), "bf16", None, False, 0.125),
    (2, 3, 257, 1032, 64, (1, 3), "bf16", [1032, 129], False, 0.125),       # nine key steps, ragged on both sides
    (3, 2, 700, 704, 64, (3, 1), "bf16", [704, 1, 640], True, 0.125),
    (8, 40, 300, 512, 64, (1, 40), "bf16", None, False, 0.125),             # more items than two per SM: persistent
    (8, 40, 600, 600, 64, (1, 1), "bf16", None, True, 0.125),               # persistent, complementary slabs
    (2, 2, 200, 328, 64, (2, 2), "bf16", None, False, -0.2),
    (2, 2, 130, 301, 64, (1, 2), "bf16", None, False, 0.125),               # rows begin at every second byte
    (1, 1, 129, 33, 64, (1, 1), "bf16", None, False, 0.125),                # the rows end within a group of eight
    (3, 5, 257, 517, 64, (3, 5), "bf16", [517, 3, 400], True, 0.125),
    (2, 3, 700, 131, 64, (2, 1), "bf16", None, False, -0.2),
    (9, 20, 401, 203, 64, (1, 20), "bf16", None, True, 0.125),              # persistent
    (9, 20, 301, 130, 64, (1, 1), "bf16", None, False, 0.125),
    (2, 3, 257, 519, 128, (1, 3), "bf16", [519, 65], False, 0.1),           # d = 128
    (3, 5, 260, 1001, 128, (3, 5), "bf16", None, True, 0.1),
    (9, 20, 301, 131, 128, (1, 20), "bf16", None, False, 0.1),              # several items a CTA
    (1, 2, 9, 30, 128, (1, 2), "bf16", None, False, 0.1),                   # too small for it
    (2, 2, 130, 302, 128, (2, 1), "bf16", [302, 77], True, 0.1),
    (2, 3, 257, 520, 128, (1, 3), "bf16", [520, 65], False, 0.1),            # d = 128, staged: nine steps of 64 keys
    (3, 2, 700, 704, 128, (3, 1), "bf16", [704, 1, 640], True, 0.1),
    (2, 2, 200, 328, 128, (2, 2), "bf16", None, False, -0.2),
    (1, 1, 1, 8, 128, (1, 1), "bf16", None, False, 0.1),
    (1, 2, 70, 131, 64, (1, 2), "f32", None, False, 0.125),
    (1, 2, 300, 130, 128, (1, 1), "f32", None, False, 0.1),
    (1, 1, 1, 1, 64, (1, 1), "bf16", None, False, 1.0),
    (2, 2, 100, 31, 64, (1, 2), "bf16", [31, 5], False, 0.125),             # few values to a row: read one by one ...
    (2, 2, 256, 63, 64, (1, 2), "bf16", None, True, -0.2),
    (2, 2, 257, 63, 64, (2, 1), "bf16", [63, 1], False, 0.125),             # ... staged
    (1, 2, 100, 65, 64, (1, 2), "bf16", None, True, 0.125),
    (2, 2, 100, 31, 128, (1, 2), "bf16", [31, 5], True, 0.1),
]


@pytest.mark.parametrize("case", CASES, ids=[str(c[:5]) + c[6] for c in CASES])
def test_bias_edges(case):
    from paper_2107_06419_b200 import api
    B, H, Nq, Nk, d, (bb, hb), kind, valid, causal, scale = case
    rng = np.random.default_rng(Nq + Nk)
    Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, d)), rand_bits(rng, (B, H, Nk, d)), rand_bits(rng, (B, H, Nk, d))
    bias = (2.0 * rng.standard_normal((bb, hb, Nq, Nk))).astype(np.float32)
    if Nk > 8:
        bias[rng.random(bias.shape) < 0.02] = -np.inf
        bias[:, :, Nq // 2] = -np.inf                                       # a row that sees nothing
        bias[:, :, :, :min(Nk - 1, 128)][:, :, ::3] = -np.inf                # rows whose first key tile is switched off
    bits = inputs.f32_to_bf16_bits(np.where(np.isinf(bias), 0, bias)).reshape(bias.shape)
    exact = np.where(np.isinf(bias), -np.inf, inputs.bf16_bits_to_f32(bits).reshape(bias.shape)) if kind == "bf16" else bias
    bt = torch.from_numpy(exact.astype(np.float32)).to(torch.bfloat16 if kind == "bf16" else torch.float32).cuda()
    vl = None if valid is None else np.array(valid, dtype=np.int32)
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = oracle.attention(Qb, Kb, Vb, scale, valid_len=vl, causal=causal, bias=np.broadcast_to(exact, (B, H, Nq, Nk)), want_lse=True)
    live = np.isfinite(ref["LSE"])
    for want_lse in (False, True):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda") if want_lse else None
        api.flat_attn_fwd_ex(Q, K, V, O, scale, k_valid_len=None if vl is None else torch.from_numpy(vl).cuda(), status=status,
                             causal=causal, lse=lse, bias=bt)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got = bf16_to_f64(O)
        check_bf16(got, ref["O"], "bias")
        assert np.all(got[~live] == 0.0)
        if want_lse:
            lg = lse.cpu().numpy()
            assert np.all(np.isneginf(lg[~live])) and np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)
