"""Packed batches of sequences of one length (dealt to the SMs in advance) against the oracle, and, at d = 128, bit for bit against
each sequence by itself; batches that only look alike (keys of other lengths)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu


def call(api, Q, K, V, cq, ck, longest, causal):
    O = torch.full_like(Q, float("nan"))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    as_t = lambda x: torch.from_numpy(np.asarray(x, dtype=np.int32)).cuda()
    api.flat_attn_varlen_fwd(Q, K, V, O, as_t(cq), as_t(ck), longest, Q.shape[2] ** -0.5, causal=causal, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return O


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("N", [1, 63, 64, 65, 128, 129, 256, 257, 513])
def test_one_length(N, causal, d):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(N + d)
    seqs, H = 80, 6                                      # 480 items a slab: three to four per SM
    Qb, Kb, Vb = (rand_bits(rng, (seqs * N, H, d)) for _ in range(3))
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    cu = np.arange(seqs + 1) * N
    O = call(api, Q, K, V, cu, cu, N, causal)
    assert torch.equal(O, call(api, Q, K, V, cu, cu, N, causal))
    for s in (0, 37, seqs - 1) if d == 128 else ():      # (d = 64: a CTA's reference maximum goes on from item to item)
        at = slice(s * N, (s + 1) * N)
        assert torch.equal(O[at], call(api, Q[at], K[at], V[at], [0, N], [0, N], N, causal))
    ref = oracle.attention_varlen(Qb, Kb, Vb, cu.astype(np.int32), cu.astype(np.int32), d ** -0.5, causal=causal)
    check_bf16(bf16_to_f64(O), ref, "one length")


@pytest.mark.parametrize("d", [64, 128])
def test_keys_of_other_lengths(d):
    """As many keys as queries in all, but not in every sequence (one has none)."""
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(d)
    seqs, H, N = 80, 6, 100
    lk = np.full(seqs, N)
    lk[0::2] -= 40
    lk[1::2] += 40
    lk[2], lk[3] = 0, 200
    cq, ck = np.arange(seqs + 1) * N, np.concatenate([[0], np.cumsum(lk)])
    assert ck[-1] == cq[-1]
    Qb, Kb, Vb = (rand_bits(rng, (seqs * N, H, d)) for _ in range(3))
    O = call(api, bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb), cq, ck, N, False)
    ref = oracle.attention_varlen(Qb, Kb, Vb, cq.astype(np.int32), ck.astype(np.int32), d ** -0.5)
    check_bf16(bf16_to_f64(O), ref, "keys of other lengths")
