"""A packed call whose sequence offsets are written by the kernel right before it on the stream, one that lets its successor start
early (the library's normalisation layer, gamma = 0: every row of its output is beta, here the bits of the offsets)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def lengths(form, rng):
    if form == "slots":                                  # too many units to sort, a long sequence: one CTA per slot, most of them empty
        n = rng.integers(1, 31, 1020)
        n[rng.integers(0, 1020)] = 1800
        return n
    if form == "equal":
        return np.full(24, int(rng.integers(150, 500)))
    return rng.integers(1, 1200, 24)                     # sorted


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("form", ["slots", "equal", "sorted"])
def test_offsets_from_the_kernel_before(form, causal, d):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(11)
    H, rows = 2, 60000
    seqs = len(lengths(form, rng))
    D = -(-2 * (seqs + 1) // 8) * 8
    X = torch.randn(rows, D, device="cuda").to(torch.bfloat16)
    gamma = torch.zeros(D, dtype=torch.bfloat16, device="cuda")
    Y = torch.zeros_like(X)
    cu = Y[-1].view(torch.int32)[:seqs + 1]              # the last row: written when the launch is nearly over
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(12):
        n = lengths(form, rng)
        off = np.concatenate([[0], np.cumsum(n)]).astype(np.int32)
        assert off[-1] < 0x7f80                          # (bf16 numbers, none of them a NaN or -0)
        total = int(off[-1])
        bits = np.zeros(D // 2, dtype=np.int32)
        bits[:seqs + 1] = off
        beta = torch.from_numpy(bits).cuda().view(torch.bfloat16)
        Q, K, V = (torch.randn(total, H, d, device="cuda").to(torch.bfloat16) for _ in range(3))
        O, want = torch.full_like(Q, float("nan")), torch.full_like(Q, float("nan"))
        torch.cuda.synchronize()
        api.flat_layernorm_fwd(X, gamma, beta, Y)
        api.flat_attn_varlen_fwd(Q, K, V, O, cu, cu, int(n.max()), d ** -0.5, causal=causal, status=status)
        torch.cuda.synchronize()
        assert np.array_equal(cu.cpu().numpy(), off)
        there = torch.from_numpy(off).cuda()
        torch.cuda.synchronize()
        api.flat_attn_varlen_fwd(Q, K, V, want, there, there, int(n.max()), d ** -0.5, causal=causal, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and torch.isfinite(want).all()
        assert torch.equal(O, want)
