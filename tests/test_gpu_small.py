"""The small-head kernel (bf16, d = 16 and 32) against the oracle at the edges of its tiles (128 queries, 96 keys, four ring stages)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2107_06419_b200 import inputs
from helpers import bf16_tensor, bf16_to_f64, rand_bits

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, Nq, Nk, d, masked, causal, sigma
    (1, 1, 1, 1, 16, False, False, 1.0),
    (1, 2, 127, 95, 32, False, False, 1.0),
    (2, 2, 128, 96, 16, True, False, 1.0),
    (2, 3, 129, 97, 32, True, True, 1.0),
    (1, 2, 300, 481, 16, False, True, 1.0),          # five key tiles and one key: the rings wrap
    (3, 2, 257, 900, 32, True, False, 4.0),          # logits of tens: the reference maximum is overtaken
    (1, 1, 200, 70, 32, False, True, 1.0),           # the first 130 queries see no key
    (40, 16, 130, 1000, 32, False, False, 1.0),      # several CTAs per SM
]


@pytest.mark.parametrize("case", CASES, ids=[str(c) for c in CASES])
def test_small_heads(case):
    from paper_2107_06419_b200 import api
    B, H, Nq, Nk, d, masked, causal, sigma = case
    rng = np.random.default_rng(1000 * d + Nk)
    Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, d), sigma), rand_bits(rng, (B, H, Nk, d), sigma), rand_bits(rng, (B, H, Nk, d))
    vl = rng.integers(0, Nk + 1, size=B).astype(np.int32) if masked else None
    if masked:
        vl[0] = 0
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, Nq), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.flat_attn_fwd_ex(Q, K, V, O, d ** -0.5, k_valid_len=None if vl is None else torch.from_numpy(vl).cuda(),
                         status=status, causal=causal, lse=lse)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and api.flat_attn_last_variant() == api.FLAT_VARIANT_SMALL
    ref = oracle.attention(Qb, Kb, Vb, d ** -0.5, valid_len=vl, causal=causal, want_lse=True)
    got, want = bf16_to_f64(O), ref["O"]
    # O is rounded to bf16 (eight significant bits: half a step is at most 2^-8 of the value); head and remainder of a weight carry 2^-17 of it, the exponentials and fp32
    # sums less: together below 2^-15 of the largest |V|
    vmax = np.abs(inputs.bf16_bits_to_f32(Vb)).max()
    assert np.all(np.isfinite(got)) and np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -15 * vmax)
    live = np.isfinite(ref["LSE"])
    lg = lse.cpu().numpy()
    assert np.all(np.isneginf(lg[~live])) and np.all(got[~live] == 0.0)
    assert np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-4)
