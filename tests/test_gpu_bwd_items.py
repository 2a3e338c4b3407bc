"""The backward kernels with more tiles than SMs: a CTA takes over further tiles, of other lengths and of none, and its rings,
barrier phases and accumulators run on (bars of tests/test_gpu_bwd.py)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_tensor, rand_bits
from test_gpu_bwd import api, check_grad, run_fwd_bwd  # noqa: F401  (the fixture and the bars)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Nq,Nk,causal,masked", [
    (16, 32, 40, 30, False, False),                      # one short step a tile, 512 tiles
    (12, 16, 130, 300, False, True),                     # key tiles that nothing sees between others; batches without a key
    (8, 16, 420, 260, True, False),                      # query tiles that see no key, the rest from one to three steps
    (4, 16, 700, 900, True, True)])
def test_more_tiles_than_sms(api, d, B, H, Nq, Nk, causal, masked):  # noqa: F811
    rng = np.random.default_rng(Nq + Nk + d)
    Qb, Kb, Vb, dOb = (rand_bits(rng, (B, H, n, d)) for n in (Nq, Nk, Nk, Nq))
    vl = (np.arange(B) * Nk // (B - 1)).astype(np.int32) if masked else None
    O, lse, dQ, dK, dV = run_fwd_bwd(api, Qb, Kb, Vb, dOb, d ** -0.5, vl=vl, causal=causal)
    ref = oracle.attention_bwd(Qb, Kb, Vb, dOb, d ** -0.5, causal=causal, valid_len=vl)
    for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
        check_grad(got, ref[name], "%s %s" % (name, (B, H, Nq, Nk, d, causal, masked)))
        assert np.all(got[ref[name] == 0] == 0) if masked else True, name   # (what nothing sees is zero, not small)


@pytest.mark.parametrize("d", [64, 128])
def test_gradients_on_16_byte_boundaries(api, d):  # noqa: F811
    """Gradients that lie on a 16-byte but not on a 32-byte boundary are stored in halves: the same bits."""
    B, H, N = 3, 5, 200
    rng = np.random.default_rng(d)
    Q, K, V, dO = (bf16_tensor(rand_bits(rng, (B, H, N, d))) for _ in range(4))
    O, lse, delta = torch.empty_like(Q), torch.empty(B, H, N, device="cuda"), torch.empty(B, H, N, device="cuda")
    api.flat_attn_fwd_ex(Q, K, V, O, d ** -0.5, lse=lse)
    got = []
    for off in (0, 8):                                   # (elements)
        grads = [torch.full((Q.numel() + 8,), float("nan"), dtype=torch.bfloat16, device="cuda")[off:off + Q.numel()].view_as(Q)
                 for _ in range(3)]
        assert all(g.data_ptr() % 32 == 2 * off for g in grads)
        api.flat_attn_bwd_ex(Q, K, V, O, dO, lse, *grads, delta, d ** -0.5)
        got.append(torch.stack(grads).view(torch.int16).cpu())
    assert torch.equal(got[0], got[1])
