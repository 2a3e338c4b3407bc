"""The sorted deal of packed batches: sequences without queries or without keys, one-token ones, lengths at the edges of slabs and
key tiles, more items than SMs, and batches beyond the table (more than 1024 units)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("case", ["edges", "many", "beyond"])
def test_packed_deal(case, causal):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(11)
    if case == "edges":
        H, lq, lk = 3, [0, 1, 255, 256, 257, 512, 700, 5, 129], [7, 0, 255, 128, 300, 1, 900, 5, 64]
    elif case == "many":
        H, lq = 16, rng.integers(1, 700, 60)
        lk = lq
    else:
        H, lq = 1, rng.integers(1, 40, 1100)
        lk = lq
    cu_q, cu_k = (np.concatenate([[0], np.cumsum(x)]).astype(np.int32) for x in (lq, lk))
    Qb, Kb, Vb = (rand_bits(rng, (int(n), H, 64)) for n in (cu_q[-1], cu_k[-1], cu_k[-1]))
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = []
    for _ in range(2):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        api.flat_attn_varlen_fwd(Q, K, V, O, torch.from_numpy(cu_q).cuda(), torch.from_numpy(cu_k).cuda(), int(max(lq)), 0.125,
                                 causal=causal, status=status)
        out.append(O)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.equal(*out)
    check_bf16(bf16_to_f64(out[0]), oracle.attention_varlen(Qb, Kb, Vb, cu_q, cu_k, 0.125, causal=causal), case)
