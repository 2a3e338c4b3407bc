"""The two-tile kernel for head size 128 where its 64-key steps change: step counts around the two logit buffers, ragged rows and
keys, masks that give the warps of a tile different numbers of full steps, a negative scale, rising logits, lse."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nk", [1, 63, 64, 65, 127, 128, 129, 192, 193, 321, 704])
@pytest.mark.parametrize("causal", [False, True])
def test_d128_edges(Nk, causal):
    from paper_2107_06419_b200 import api
    B, H = 2, 3
    for Nq, scale, rising in ((17, 0.1, 0.0), (128, -0.2, 0.0), (257, 0.09, 0.0), (300, 0.09, 40.0)):
        rng = np.random.default_rng(Nq + Nk)
        Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, 128)), rand_bits(rng, (B, H, Nk, 128)), rand_bits(rng, (B, H, Nk, 128))
        if rising:                       # keys that grow along the sequence: the reference of the first step goes stale
            from paper_2107_06419_b200 import inputs
            grown = inputs.bf16_bits_to_f32(Kb).reshape(Kb.shape) * (1 + rising * np.arange(Nk, dtype=np.float32)[:, None] / Nk)
            Kb = inputs.f32_to_bf16_bits(grown.astype(np.float32)).reshape(Kb.shape)
        vl = np.array([Nk, max(1, Nk - 70)], dtype=np.int32)
        ref = oracle.attention(Qb, Kb, Vb, scale, valid_len=vl, causal=causal, want_lse=True)
        Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, scale, k_valid_len=torch.from_numpy(vl).cuda(), status=status, causal=causal, lse=lse,
                             variant=api.FLAT_VARIANT_TC2)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        live = np.isfinite(ref["LSE"])
        got, lg = bf16_to_f64(O), lse.cpu().numpy()
        check_bf16(got, ref["O"], "d128 Nq=%d" % Nq)
        assert np.all(got[~live] == 0.0) and np.all(np.isneginf(lg[~live]))
        assert np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)


@pytest.mark.parametrize("causal", [False, True])
def test_d128_packed_edges(causal):
    from paper_2107_06419_b200 import api
    H = 2
    lq = [1, 63, 0, 128, 129, 600, 256, 130, 128]
    lk = [64, 65, 5, 700, 129, 600, 0, 700, 701]                          # (warps of one tile end their full steps at different steps)
    cq, ck = (np.cumsum([0] + x).astype(np.int32) for x in (lq, lk))
    rng = np.random.default_rng(5)
    Qb, Kb, Vb = rand_bits(rng, (sum(lq), H, 128)), rand_bits(rng, (sum(lk), H, 128)), rand_bits(rng, (sum(lk), H, 128))
    ref = oracle.attention_varlen(Qb, Kb, Vb, cq, ck, 0.09, causal=causal)
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    first = None
    for _ in range(10):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_varlen_fwd(Q, K, V, O, torch.from_numpy(cq).cuda(), torch.from_numpy(ck).cuda(), max(lq), 0.09, causal=causal, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got = bf16_to_f64(O)
        check_bf16(got, ref, "packed d128")
        assert first is None or np.array_equal(got, first)
        first = got


@pytest.mark.parametrize("case", [(19, 20, 300, 1, False), (10, 16, 257, 64, False), (10, 16, 256, 130, False), (5, 31, 300, 200, True),
                                  (13, 12, 100, 333, True)], ids=str)
def test_d128_several_items_per_cta(case):
    """More items than SMs: CTAs take several in turn (with one, two and more key steps; rows without keys under the causal mask)."""
    from paper_2107_06419_b200 import api
    B, H, Nq, Nk, causal = case
    rng = np.random.default_rng(Nq + Nk)
    Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, 128)), rand_bits(rng, (B, H, Nk, 128)), rand_bits(rng, (B, H, Nk, 128))
    ref = oracle.attention(Qb, Kb, Vb, 0.09, causal=causal, want_lse=True)
    live = np.isfinite(ref["LSE"])
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    for _ in range(3):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, 0.09, status=status, causal=causal, lse=lse)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got, lg = bf16_to_f64(O), lse.cpu().numpy()
        check_bf16(got, ref["O"], "several items")
        assert np.all(got[~live] == 0.0) and np.all(np.isneginf(lg[~live])) and np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)
