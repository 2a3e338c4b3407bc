"""Head size 128, more items than SMs: a CTA takes over items of other lengths and of none, with their bias tiles, or has several of one
length dealt to it; and one item a CTA over many keys."""
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


@pytest.mark.parametrize("Nk", [200, 203])                                # (rows of the bias on 16-byte boundaries; at any)
@pytest.mark.parametrize("B,H,Nq,causal", [(40, 8, 30, False), (20, 8, 270, True), (11, 16, 257, False)])
def test_key_counts_with_bias(B, H, Nq, Nk, causal):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(Nq + Nk)
    Qb, Kb, Vb = (rand_bits(rng, (B, H, n, 128)) for n in (Nq, Nk, Nk))
    vl = (np.arange(B) * Nk // (B - 1)).astype(np.int32)                  # from none to all
    vl[1::5] = 0                                                          # (and none between others)
    bias = rand_bits(rng, (1, H, Nq, Nk), 2.0)
    ref = oracle.attention(Qb, Kb, Vb, 0.09, valid_len=vl, causal=causal, bias=bias, want_lse=True)
    live = np.isfinite(ref["LSE"])
    Q, K, V, bt, vlt = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb), bf16_tensor(bias), torch.from_numpy(vl).cuda()
    first = None
    for _ in range(3):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, H, Nq), float("nan"), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, 0.09, k_valid_len=vlt, status=status, causal=causal, lse=lse, bias=bt)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got, lg = bf16_to_f64(O), lse.cpu().numpy()
        check_bf16(got, ref["O"], "key counts, bias")
        assert np.all(got[~live] == 0.0) and np.all(np.isneginf(lg[~live])) and np.all(np.abs(lg[live] - ref["LSE"][live]) <= 1e-3)
        assert first is None or np.array_equal(got, first)
        first = got


# Items that weigh the same, on both sides of the lines between dealing them, taking them over and one a CTA (three keys a query; 1024
# keys; bias rows to be shifted, 256 keys)
@pytest.mark.parametrize("bias", [False, True])
@pytest.mark.parametrize("B,H,Nq,Nk", [(50, 8, 20, 60), (50, 8, 20, 61), (19, 8, 10, 30), (40, 8, 300, 290), (9, 8, 600, 1024), (9, 8, 600, 1025),
                                      (10, 8, 300, 255), (10, 8, 300, 257)])
def test_equal_items(B, H, Nq, Nk, bias):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(Nq + Nk)
    Qb, Kb, Vb = (rand_bits(rng, (B, H, n, 128)) for n in (Nq, Nk, Nk))
    bb = rand_bits(rng, (1, H, Nq, Nk)) if bias else None
    rows = np.unique(np.concatenate([np.arange(B * H) * Nq + at for at in (0, Nq // 2, Nq - 1)])).astype(np.int64)   # (of every item)
    ref = oracle.attention(Qb, Kb, Vb, 0.09, rows=rows, bias=bb)["O"]
    O = torch.full((B, H, Nq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.flat_attn_fwd_ex(bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb), O, 0.09, status=status,
                         bias=bf16_tensor(bb) if bias else None, variant=api.FLAT_VARIANT_TC2)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = bf16_to_f64(O)
    assert np.all(np.isfinite(got))
    check_bf16(got.reshape(-1, 128)[rows], ref, "equal items")


@pytest.mark.parametrize("causal", [False, True])
def test_one_item_and_many_keys(causal):
    """No more items than SMs, more than 8192 keys."""
    from paper_2107_06419_b200 import api
    B, H, Nq, Nk = 3, 2, 300, 8500
    rng = np.random.default_rng(7)
    Qb, Kb, Vb = (rand_bits(rng, (B, H, n, 128)) for n in (Nq, Nk, Nk))
    vl = np.array([Nk, 0, 8300], dtype=np.int32)
    ref = oracle.attention(Qb, Kb, Vb, 0.09, valid_len=vl, causal=causal)
    O = torch.full((B, H, Nq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.flat_attn_fwd_ex(bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb), O, 0.09, k_valid_len=torch.from_numpy(vl).cuda(),
                         status=status, causal=causal, variant=api.FLAT_VARIANT_TC2)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = bf16_to_f64(O)
    check_bf16(got, ref["O"], "many keys")
    assert np.all(got[1] == 0.0)


def test_while_another_stream_holds_sms():
    """CTAs of the launch start late, and a question may find none while some have not started: the bits of an undisturbed launch."""
    from paper_2107_06419_b200 import api
    g = torch.Generator(device="cuda").manual_seed(3)
    B, H, N = 8, 16, 700
    Q, K, V = (torch.randn(B, H, N, 128, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(3))
    W = torch.randn(4096, 4096, device="cuda", dtype=torch.bfloat16, generator=g)
    vl = torch.randint(0, N + 1, (B,), device="cuda", generator=g, dtype=torch.int32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    forms = [dict(k_valid_len=vl), dict(causal=True), dict()]             # (taken over twice, dealt)
    alone = []
    for kw in forms:
        alone.append(torch.empty_like(Q))
        api.flat_attn_fwd_ex(Q, K, V, alone[-1], 0.09, status=status, **kw)
    torch.cuda.synchronize()
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    outs = []
    for i in range(12):
        with torch.cuda.stream(other):
            for _ in range(2):
                torch.matmul(W, W)
        O = torch.full_like(Q, float("nan"))
        own.wait_stream(torch.cuda.current_stream())
        api.flat_attn_fwd_ex(Q, K, V, O, 0.09, status=status, stream=own.cuda_stream, **forms[i % 3])
        outs.append(O)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, O in enumerate(outs):
        assert torch.equal(O.view(torch.int16), alone[i % 3].view(torch.int16)), i
