"""The kernel for a few queries per head (bf16, d = 64 and 128) against the oracle: one to sixteen queries, shares of the keys
that are empty, ragged or longer than the ring, masks on both sides."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, Nq, Nk, d, valid lengths, causal, sigma
    (1, 1, 1, 1, 128, None, False, 1.0),
    (1, 2, 1, 63, 64, None, False, 1.0),
    (2, 2, 8, 129, 128, [129, 0], False, 1.0),
    (3, 2, 9, 700, 64, [700, 1, 65], True, 1.0),
    (2, 3, 16, 1500, 128, [1500, 64], True, 1.0),
    (2, 2, 5, 5000, 64, [5000, 4097], False, 4.0),           # several turns of the ring; logits of tens
    (4, 40, 1, 3000, 128, [3000, 750, 2049, 1], False, 1.0),
    (1, 4, 2, 20000, 128, None, True, 1.0),                  # few heads: the widest split
    (1, 1, 16, 10, 64, None, True, 1.0),                     # the first six queries see no key
    (300, 3, 3, 100, 64, None, False, 1.0),                  # many short heads
]


@pytest.mark.parametrize("case", CASES, ids=[str(c[:5]) for c in CASES])
def test_decode(case):
    from paper_2107_06419_b200 import api
    B, H, Nq, Nk, d, valid, causal, sigma = case
    rng = np.random.default_rng(Nk + d)
    Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, d), sigma), rand_bits(rng, (B, H, Nk, d), sigma), rand_bits(rng, (B, H, Nk, d))
    vl = None if valid is None else np.array(valid, dtype=np.int32)
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = []
    for _ in range(2):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, d ** -0.5, k_valid_len=None if vl is None else torch.from_numpy(vl).cuda(),
                             status=status, causal=causal, lse=lse)
        assert api.flat_attn_last_variant() == api.FLAT_VARIANT_DECODE
        out.append((O, lse))
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and all(torch.equal(a, b) for a, b in zip(*out))
    ref = oracle.attention(Qb, Kb, Vb, d ** -0.5, valid_len=vl, causal=causal, want_lse=True)
    got, lg = bf16_to_f64(out[0][0]), out[0][1].cpu().numpy()
    check_bf16(got, ref["O"], "decode")
    live = np.isfinite(ref["LSE"])
    assert np.all(np.isneginf(lg[~live])) and np.all(got[~live] == 0.0)
    assert np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)
