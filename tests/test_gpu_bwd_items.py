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


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_many_steps_a_tile(api, d, causal):  # noqa: F811
    """Tiles of up to twelve steps, so that the next one is asked for in the middle of a tile, more of them than SMs."""
    B, H, N = 2, 8, 1500
    rng = np.random.default_rng(d + causal)
    Qb, Kb, Vb, dOb = (rand_bits(rng, (B, H, N, d)) for _ in range(4))
    O, lse, dQ, dK, dV = run_fwd_bwd(api, Qb, Kb, Vb, dOb, d ** -0.5, causal=causal)
    heads = [0, 3, 7, 8, 12, 15]
    ref = oracle.attention_bwd(Qb, Kb, Vb, dOb, d ** -0.5, causal=causal, heads=heads)
    for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
        assert np.all(np.isfinite(got)), name
        check_grad(got.reshape(B * H, N, d)[heads], ref[name], "%s d=%d causal=%s" % (name, d, causal))


def test_groups_of_heads(api):  # noqa: F811
    """Under the causal mask the tiles of as many heads as fit L2 go together: 62 heads here, and the other eight."""
    B, H, N, d = 5, 14, 1500, 128
    rng = np.random.default_rng(9)
    Qb, Kb, Vb, dOb = (rand_bits(rng, (B, H, N, d)) for _ in range(4))
    vl = np.array([1500, 700, 0, 1499, 1300], dtype=np.int32)
    O, lse, dQ, dK, dV = run_fwd_bwd(api, Qb, Kb, Vb, dOb, d ** -0.5, vl=vl, causal=True)
    heads = [0, 20, 56, 61, 62, 69]
    ref = oracle.attention_bwd(Qb, Kb, Vb, dOb, d ** -0.5, causal=True, valid_len=vl, heads=heads)
    for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
        assert np.all(np.isfinite(got)) and np.all(got[2] == 0), name
        check_grad(got.reshape(B * H, N, d)[heads], ref[name], "%s, groups of heads" % name)


@pytest.mark.parametrize("d", [64, 128])
def test_while_another_stream_holds_sms(api, d):  # noqa: F811
    """CTAs of a launch start late, and a question may find none while some have not started: the bits of an undisturbed call."""
    g = torch.Generator(device="cuda").manual_seed(d)
    B, H, N = 4, 16, 900
    Q, K, V, dO = (torch.randn(B, H, N, d, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(4))
    W = torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16, generator=g)
    O, lse = torch.empty_like(Q), torch.empty(B, H, N, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    for causal in (False, True):
        api.flat_attn_fwd_ex(Q, K, V, O, d ** -0.5, lse=lse, causal=causal)
        calls = []
        for i in range(7):
            grads = [torch.full_like(Q, float("nan")) for _ in range(3)]
            delta = torch.empty_like(lse)
            own.wait_stream(torch.cuda.current_stream())
            if i > 0:                                    # (the first one alone)
                with torch.cuda.stream(other):
                    for _ in range(2):
                        torch.matmul(W, W)
            api.flat_attn_bwd_ex(Q, K, V, O, dO, lse, *grads, delta, d ** -0.5, status=status, causal=causal, stream=own.cuda_stream)
            if i == 0:
                torch.cuda.synchronize()
            calls.append((grads, delta))
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        for grads, delta in calls[1:]:
            assert torch.equal(delta, calls[0][1])
            assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(grads, calls[0][0]))
