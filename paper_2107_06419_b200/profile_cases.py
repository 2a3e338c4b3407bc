"""One named case of the library, a few launches, for profiler captures (ncu) and quick timings.

    python -m paper_2107_06419_b200.profile_cases CASE [--workload NAME] [--launches N]

CASE: fused | fused_lse | naive | backward | fp32 | bias | layernorm | layer.  The workload is one of
`inputs.WORKLOADS` (default p_4k_small, a quarter of c2: inputs larger than L2, a few hundred MB on the
device); inputs are the seeded generator's.  Prints the mean launch time from CUDA events.  `fp32` runs the
split-tf32 tensor-core kernel (`--variant 1`: the FFMA kernel).
Cases with sizes of their own, on random inputs: decode (B16 H16 1 x 8192, d 128, 25-100 % of the cache filled) | small (B64 H8
1000^2, d 32) | packed (32 sequences of 40 to 2000 tokens, 12 heads, d 64) | fp32_d128 (B2 H16 4096^2) | fc (512 x 3072 -> 768).
"""
from __future__ import annotations

import argparse

import numpy as np
import torch

from . import api, inputs


def _normal(*shape, dtype=torch.bfloat16):
    return torch.randn(*shape, device="cuda", dtype=torch.float32).to(dtype)


def _attention(B, H, Nq, Nk, d, dtype=torch.bfloat16, filled=None):
    torch.manual_seed(1)
    Q, K, V = (_normal(B, H, n, d, dtype=dtype) for n in (Nq, Nk, Nk))
    O, status = torch.empty_like(Q), torch.zeros(1, dtype=torch.int32, device="cuda")
    vl = None if filled is None else torch.randint(int(filled * Nk), Nk + 1, (B,), device="cuda", dtype=torch.int32)
    keys = B * Nk if vl is None else int(vl.sum())
    return (lambda: api.flat_attn_fwd_ex(Q, K, V, O, d ** -0.5, k_valid_len=vl, status=status)), 4.0 * H * Nq * keys * d, status


def _packed():
    torch.manual_seed(1)
    H, d = 12, 64
    lens = [int(round(40 * 50 ** (i / 31.0))) for i in range(32)]
    lens = [lens[(7 * i) % 32] for i in range(32)]
    Q, K, V = (_normal(sum(lens), H, d) for _ in range(3))
    O, status = torch.empty_like(Q), torch.zeros(1, dtype=torch.int32, device="cuda")
    cu = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32).cuda()
    step = lambda: api.flat_attn_varlen_fwd(Q, K, V, O, cu, cu, max(lens), d ** -0.5, status=status)
    return step, 4.0 * H * d * sum(n * n for n in lens), status


def _fc():
    X, W, Y = _normal(512, 3072), _normal(768, 3072), _normal(512, 768)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    return (lambda: api.flat_fc_fwd(X, W, Y, status=status)), 2.0 * 512 * 3072 * 768, status


# case -> (step, floating-point operations, status word), with sizes of its own
OWN = {"decode": lambda: _attention(16, 16, 1, 8192, 128, filled=0.25), "small": lambda: _attention(64, 8, 1000, 1000, 32),
       "fp32_d128": lambda: _attention(2, 16, 4096, 4096, 128, torch.float32), "packed": _packed, "fc": _fc}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("case", choices=["fused", "fused_lse", "naive", "backward", "fp32", "bias", "layernorm", "layer"] + sorted(OWN))
    ap.add_argument("--workload", default="p_4k_small")
    ap.add_argument("--launches", type=int, default=4)
    ap.add_argument("--variant", type=int, default=0)
    args = ap.parse_args()
    if args.case in OWN:
        return run(args.case, "its own sizes", *OWN[args.case](), args.launches)
    w = inputs.WORKLOADS[args.workload]
    dev = torch.device("cuda")
    Qb, Kb, Vb = inputs.make_qkv_bf16(w)
    t = lambda bits: torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).to(dev)
    Q, K, V = t(Qb), t(Kb), t(Vb)
    O = torch.empty_like(Q)
    vl = torch.from_numpy(inputs.make_valid_len(w)).to(dev) if w.masked else None
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    flops = float(w.flops)
    if args.case == "fused":
        step = lambda: api.flat_attn_fwd_ex(Q, K, V, O, w.scale, k_valid_len=vl, status=status, variant=args.variant)
    elif args.case == "fused_lse":
        lse = torch.empty((w.B, w.H, w.Nq), dtype=torch.float32, device=dev)
        step = lambda: api.flat_attn_fwd_ex(Q, K, V, O, w.scale, k_valid_len=vl, status=status, variant=args.variant, lse=lse)
    elif args.case == "naive":
        L = torch.empty((w.B, w.H, w.Nq, w.Nk), dtype=torch.float32, device=dev)
        A = torch.empty((w.B, w.H, w.Nq, w.Nk), dtype=torch.bfloat16, device=dev)
        step = lambda: api.flat_attn_naive_fwd_ex(Q, K, V, O, L, A, w.scale, k_valid_len=vl)
    elif args.case == "backward":
        dO = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 5, 0, Qb.size)).reshape(Qb.shape))
        lse = torch.empty((w.B, w.H, w.Nq), dtype=torch.float32, device=dev)
        delta = torch.empty_like(lse)
        dQ, dK, dV = torch.empty_like(Q), torch.empty_like(K), torch.empty_like(K)
        api.flat_attn_fwd_ex(Q, K, V, O, w.scale, k_valid_len=vl, status=status, lse=lse)
        step = lambda: api.flat_attn_bwd_ex(Q, K, V, O, dO, lse, dQ, dK, dV, delta, w.scale, k_valid_len=vl, status=status)
        flops *= 2.5
    elif args.case == "fp32":
        Qf, Kf, Vf = Q.float(), K.float(), V.float()
        Of = torch.empty_like(Qf)
        step = lambda: api.flat_attn_fwd_ex(Qf, Kf, Vf, Of, w.scale, k_valid_len=vl, status=status, variant=args.variant)
    elif args.case == "bias":
        bias = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 6, 0, w.H * w.Nq * w.Nk)).reshape(1, w.H, w.Nq, w.Nk))
        step = lambda: api.flat_attn_fwd_ex(Q, K, V, O, w.scale, k_valid_len=vl, status=status, bias=bias)
    elif args.case == "layernorm":
        # the token-major activations of the workload's layer: [B * Nq, H * d]
        X = Q.view(w.B * w.Nq, w.H * w.d)
        R = torch.empty_like(X).copy_(K.view(-1)[:X.numel()].view_as(X)) if K.numel() >= X.numel() else torch.zeros_like(X)
        Y = torch.empty_like(X)
        g = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 7, 0, w.H * w.d)))
        b = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 8, 0, w.H * w.d)))
        step = lambda: api.flat_layernorm_fwd(X, g, b, Y, residual=R)
        flops = 0.0
    else:  # layer
        Dm = w.H * w.d
        X = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 9, 0, w.B * w.Nq * Dm)).reshape(w.B, w.Nq, Dm))
        Wqkv = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 10, 0, 3 * Dm * Dm) * np.float32(Dm ** -0.5)).reshape(3 * Dm, Dm))
        Wo = t(inputs.f32_to_bf16_bits(inputs.normal_f32(inputs.DEFAULT_SEED, 11, 0, Dm * Dm) * np.float32(Dm ** -0.5)).reshape(Dm, Dm))
        Y = torch.empty_like(X)
        Kl, Vl, Ol = torch.empty_like(Q), torch.empty_like(Q), torch.empty_like(Q)
        step = lambda: api.flat_attn_layer_fwd(X, Wqkv, Wo, Y, Q, Kl, Vl, Ol, w.scale, status=status)
        flops += 2.0 * w.B * w.Nq * Dm * 4 * Dm
    run(args.case, w.name, step, flops, status, args.launches)


def run(case, workload, step, flops, status, launches):
    step()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(launches):
        step()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / launches
    code = int(status.item())
    print("%s on %s: %.4f ms per call%s, device status %d" % (
        case, workload, ms, (", %.1f TFLOP/s" % (flops / ms / 1e9)) if flops else "", code))
    assert code == 0


if __name__ == "__main__":
    main()
