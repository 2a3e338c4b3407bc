"""Head size 128, more items than SMs with key counts: a CTA takes over items of other lengths and of none (and their bias tiles)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Nq,Nk,causal", [(40, 8, 30, 200, False), (20, 8, 270, 190, True), (11, 16, 257, 700, False)])
def test_key_counts(B, H, Nq, Nk, causal):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(Nq + Nk)
    Qb, Kb, Vb = (rand_bits(rng, (B, H, n, 128)) for n in (Nq, Nk, Nk))
    vl = (np.arange(B) * Nk // (B - 1)).astype(np.int32)                  # from none to all
    ref = oracle.attention(Qb, Kb, Vb, 0.09, valid_len=vl, causal=causal, want_lse=True)
    live = np.isfinite(ref["LSE"])
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    first = None
    for _ in range(3):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, 0.09, k_valid_len=torch.from_numpy(vl).cuda(), status=status, causal=causal, lse=lse)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got, lg = bf16_to_f64(O), lse.cpu().numpy()
        check_bf16(got, ref["O"], "key counts")
        assert np.all(got[~live] == 0.0) and np.all(np.isneginf(lg[~live])) and np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)
        assert first is None or np.array_equal(got, first)                # (whichever CTA takes an item)
        first = got
