"""The attention work that the library is measured on: what its users call, over the sizes they call it with.

Every case names a `kind` (which entry points one pass goes through) and its sizes:

  attention   flat_attn_fwd / flat_attn_fwd_ex on dense tensors: inference of encoders, decoders (causal prefill and
              decode against a partly filled key/value cache) and cross-attention over padded memories
  bias        the same with an additive [1, H, Nq, Nk] bf16 bias of the relative position, shared by the batch (T5, TrXL)
  packed      flat_attn_varlen_fwd on a batch of sequences of different lengths without padding
  training    forward with the row log-sum-exp, then flat_attn_bwd_ex
  block       an encoder block: projections and attention (flat_attn_layer_fwd), residual and normalisation, the two
              fully connected operators, residual and normalisation

The named sizes are those of the library's workloads (paper_2107_06419_b200/inputs.py) or generic ones.
"""
import math
import random

import torch

from paper_2107_06419_b200 import api


def listed():
    return [
        # One BERT-base sequence: the smallest call that is made in earnest; latency, host time and launches count.
        {"name": "bert_base_512", "kind": "attention", "B": 1, "H": 12, "Nq": 512, "Nk": 512, "d": 64},
        # A batch of BERT-large layers at 4096 tokens: the library's headline workload.
        {"name": "bert_large_4k", "kind": "attention", "B": 16, "H": 16, "Nq": 4096, "Nk": 4096, "d": 64},
        # Decoder queries over encoder memories that are padded to one length.
        {"name": "cross_masked_16k", "kind": "attention", "B": 8, "H": 12, "Nq": 1024, "Nk": 16384, "d": 64, "filled": 0.5},
        # A decoder's prompt at the longest context, head size 128: the largest call.
        {"name": "prefill_64k_d128", "kind": "attention", "B": 1, "H": 8, "Nq": 65536, "Nk": 65536, "d": 128, "causal": True},
        # A decode step: one new token per sequence against caches of different fill.
        {"name": "decode_8k_d128", "kind": "attention", "B": 16, "H": 16, "Nq": 1, "Nk": 8192, "d": 128, "filled": 0.25},
        # Small heads (head size 32), at a length that no tile divides.
        {"name": "small_heads_d32", "kind": "attention", "B": 16, "H": 8, "Nq": 1000, "Nk": 1000, "d": 32},
        # fp32 tensors, for users who need fp32 results.
        {"name": "fp32_4k", "kind": "attention", "B": 2, "H": 16, "Nq": 4096, "Nk": 4096, "d": 64, "fp32": True},
        # T5-style encoder: relative-position bias shared by the batch.
        {"name": "t5_bias_1k", "kind": "bias", "B": 8, "H": 16, "Nq": 1024, "Nk": 1024, "d": 64},
        # Serving a mix of short and long sequences, packed.
        {"name": "packed_mix_d64", "kind": "packed", "seqs": 32, "H": 12, "shortest": 40, "longest": 2000, "mix": 1, "d": 64},
        # Training step of an encoder layer at 4096 tokens.
        {"name": "train_4k_d64", "kind": "training", "B": 4, "H": 16, "Nq": 4096, "Nk": 4096, "d": 64},
        # Training step of a decoder layer, head size 128, at a length that no tile divides.
        {"name": "train_causal_3k_d128", "kind": "training", "B": 2, "H": 16, "Nq": 3000, "Nk": 3000, "d": 128, "causal": True},
        # One BERT-base encoder block on one sequence: several small operators in a row.
        {"name": "block_bert_base_512", "kind": "block", "B": 1, "H": 12, "Nq": 512, "Nk": 512, "d": 64},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _smaller(case, most):
    """The case with fewer heads, batches or tokens until its floating-point work is at most `most`."""
    while work(case)["flops"] > most:
        for key, least in (("B", 1), ("seqs", 2), ("H", 4), ("Nq", 1), ("longest", 256)):
            if case.get(key, 0) > least:
                case[key] = max(least, case[key] // 2)
                if key == "Nq":
                    case["Nk"] = max(case["Nk"] // 2, 1)
                if key == "longest":
                    case["shortest"] = min(case["shortest"], case[key])
                break
        else:
            return case
    return case


def draw(rng):
    """One more case: a use, and sizes over the range in which it is used.

    The bounds on the work keep a drawn case within the time of the largest listed one; they are lower for the
    directions and types that cost more per operation.
    """
    use = rng.choice(("encoder", "encoder", "cross", "prefill", "decode", "small heads", "fp32", "bias", "packed",
                      "training", "training", "block"))
    H = rng.choice((4, 6, 8, 12, 16, 20, 32))
    if use == "encoder":
        n = _log(rng, 64, 16384)
        return _smaller({"kind": "attention", "B": _log(rng, 1, 32), "H": H, "Nq": n, "Nk": n, "d": rng.choice((64, 128))}, 4e12)
    if use == "cross":
        return _smaller({"kind": "attention", "B": _log(rng, 1, 16), "H": H, "Nq": _log(rng, 64, 4096),
                         "Nk": _log(rng, 256, 32768), "d": rng.choice((64, 128)), "filled": 0.5}, 4e12)
    if use == "prefill":
        n = _log(rng, 256, 65536)
        return _smaller({"kind": "attention", "B": _log(rng, 1, 8), "H": H, "Nq": n, "Nk": n, "d": rng.choice((64, 128)),
                         "causal": True}, 4e12)
    if use == "decode":
        return {"kind": "attention", "B": _log(rng, 1, 32), "H": H, "Nq": rng.choice((1, 1, 1, 2, 4, 8)),
                "Nk": _log(rng, 512, 32768), "d": rng.choice((64, 128)), "filled": 0.25}
    if use == "small heads":
        n = _log(rng, 128, 4096)
        return _smaller({"kind": "attention", "B": _log(rng, 1, 32), "H": H, "Nq": n, "Nk": n, "d": rng.choice((16, 32)),
                         "causal": rng.random() < 0.3}, 1e11)
    if use == "fp32":
        n = _log(rng, 256, 8192)
        return _smaller({"kind": "attention", "B": _log(rng, 1, 8), "H": H, "Nq": n, "Nk": n, "d": rng.choice((32, 64, 64, 128)),
                         "fp32": True, "causal": rng.random() < 0.3}, 1.5e11)
    if use == "bias":
        n = _log(rng, 128, 4096)
        return _smaller({"kind": "bias", "B": _log(rng, 1, 16), "H": H, "Nq": n, "Nk": n, "d": rng.choice((64, 64, 128))}, 8e11)
    if use == "packed":
        longest = _log(rng, 256, 8192)
        return _smaller({"kind": "packed", "seqs": _log(rng, 2, 64), "H": H, "shortest": _log(rng, 16, longest),
                         "longest": longest, "mix": rng.randrange(1000), "d": rng.choice((64, 128)),
                         "causal": rng.random() < 0.5}, 3e12)
    if use == "training":
        n = _log(rng, 256, 8192)
        return _smaller({"kind": "training", "B": _log(rng, 1, 16), "H": H, "Nq": n, "Nk": n, "d": rng.choice((64, 128)),
                         "causal": rng.random() < 0.5}, 2.5e12)
    d = rng.choice((64, 128))
    n = 128 * _log(rng, 1, 32)
    return _smaller({"kind": "block", "B": _log(rng, 1, 16), "H": rng.choice((4, 8, 12, 16)), "Nq": n, "Nk": n, "d": d}, 3e12)


def _lengths(case):
    """The sequence lengths of a packed batch: over their logarithm between the shortest and the longest."""
    rng = random.Random(case["mix"])
    return [_log(rng, case["shortest"], case["longest"]) for _ in range(case["seqs"])]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, H, d = case["kind"], case["H"], case["d"]
    dtype = torch.float32 if case.get("fp32") else torch.bfloat16

    def normal(*shape, std=1.0):
        x = torch.randn(*shape, device="cuda", generator=gen, dtype=torch.float32)
        return (x * std if std != 1.0 else x).to(dtype)

    s = {"kind": kind, "scale": d ** -0.5, "causal": bool(case.get("causal"))}
    if kind == "packed":
        lens = _lengths(case)
        total = sum(lens)
        ends = torch.tensor([0] + lens, dtype=torch.int32).cumsum(0).to(torch.int32)
        s.update(Q=normal(total, H, d), K=normal(total, H, d), V=normal(total, H, d), cu=ends.cuda(), longest=max(lens))
        s["O"] = torch.empty_like(s["Q"])
        return s
    B, Nq, Nk = case["B"], case["Nq"], case["Nk"]
    if kind == "block":
        D = H * d
        s.update(X=normal(B, Nq, D), Wqkv=normal(3 * D, D, std=D ** -0.5), Wo=normal(D, D, std=D ** -0.5),
                 W1=normal(4 * D, D, std=D ** -0.5), W2=normal(D, 4 * D, std=(4 * D) ** -0.5),
                 g1=1 + normal(D, std=0.1), b1=normal(D, std=0.1), g2=1 + normal(D, std=0.1), b2=normal(D, std=0.1))
        for name in ("Q", "K", "V", "O"):
            s[name] = torch.empty(B, H, Nq, d, device="cuda", dtype=dtype)
        for name in ("attended", "normed", "Y"):
            s[name] = torch.empty_like(s["X"])
        s["wide"] = torch.empty(B, Nq, 4 * D, device="cuda", dtype=dtype)
        s["narrow"] = torch.empty_like(s["X"])
        return s
    s.update(Q=normal(B, H, Nq, d), K=normal(B, H, Nk, d), V=normal(B, H, Nk, d))
    s["O"] = torch.empty_like(s["Q"])
    s["valid"] = None
    if case.get("filled"):                              # every batch has its own number of valid keys
        least = max(1, int(case["filled"] * Nk))
        s["valid"] = torch.randint(least, Nk + 1, (B,), device="cuda", generator=gen, dtype=torch.int32)
    if kind == "bias":                                  # one learnt value per head and clipped distance
        reach = 128
        table = normal(H, 2 * reach + 1)
        at = (torch.arange(Nk, device="cuda")[None, :] - torch.arange(Nq, device="cuda")[:, None]).clamp(-reach, reach) + reach
        s["bias"] = table[:, at].reshape(1, H, Nq, Nk).contiguous()
    if kind == "training":
        s["dO"] = normal(B, H, Nq, d)
        s["lse"] = torch.empty(B, H, Nq, device="cuda", dtype=torch.float32)
        s["delta"] = torch.empty_like(s["lse"])
        s["dQ"], s["dK"], s["dV"] = torch.empty_like(s["Q"]), torch.empty_like(s["K"]), torch.empty_like(s["V"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "attention":
        if s["valid"] is None and not s["causal"] and s["Q"].dtype == torch.bfloat16:
            return api.flat_attn_fwd(s["Q"], s["K"], s["V"], s["O"], s["scale"])
        return api.flat_attn_fwd_ex(s["Q"], s["K"], s["V"], s["O"], s["scale"], k_valid_len=s["valid"], causal=s["causal"])
    if kind == "bias":
        return api.flat_attn_fwd_ex(s["Q"], s["K"], s["V"], s["O"], s["scale"], bias=s["bias"])
    if kind == "packed":
        return api.flat_attn_varlen_fwd(s["Q"], s["K"], s["V"], s["O"], s["cu"], s["cu"], s["longest"], s["scale"],
                                        causal=s["causal"])
    if kind == "training":
        api.flat_attn_fwd_ex(s["Q"], s["K"], s["V"], s["O"], s["scale"], causal=s["causal"], lse=s["lse"])
        api.flat_attn_bwd_ex(s["Q"], s["K"], s["V"], s["O"], s["dO"], s["lse"], s["dQ"], s["dK"], s["dV"], s["delta"],
                             s["scale"], causal=s["causal"])
        return {name: s[name] for name in ("O", "lse", "dQ", "dK", "dV")}
    api.flat_attn_layer_fwd(s["X"], s["Wqkv"], s["Wo"], s["attended"], s["Q"], s["K"], s["V"], s["O"], s["scale"])
    api.flat_layernorm_fwd(s["attended"], s["g1"], s["b1"], s["normed"], residual=s["X"])
    api.flat_fc_fwd(s["normed"], s["W1"], s["wide"])
    api.flat_fc_fwd(s["wide"], s["W2"], s["narrow"])
    api.flat_layernorm_fwd(s["narrow"], s["g2"], s["b2"], s["Y"], residual=s["normed"])
    return s["Y"]


def work(case):
    kind, H, d = case["kind"], case["H"], case["d"]
    size = 4 if case.get("fp32") else 2

    def visible(nq, nk):
        """The (query, key) pairs that take part."""
        if not case.get("causal"):
            return nq * nk
        return sum(min(nk, max(0, i + 1 + nk - nq)) for i in range(nq)) if nq != nk else nq * (nq + 1) // 2

    if kind == "packed":
        lens = _lengths(case)
        return {"bytes": 4 * size * H * d * sum(lens), "flops": 4 * H * d * sum(visible(n, n) for n in lens)}
    B, Nq, Nk = case["B"], case["Nq"], case["Nk"]
    rows, pairs = B * H * Nq, B * H * visible(Nq, Nk)
    if kind == "block":
        D, tokens = H * d, B * Nq
        return {"bytes": size * (2 * tokens * D + 12 * D * D), "flops": 24 * tokens * D * D + 4 * pairs * d}
    filled = (1 + case["filled"]) / 2 if case.get("filled") else 1.0   # mean share of valid keys
    keys = B * H * Nk * filled
    nbytes = size * d * (2 * rows + 2 * keys)
    if kind == "bias":
        nbytes += size * H * Nq * Nk
    if kind == "training":                              # Q, K, V, dO in; O, lse, dQ, dK, dV out
        return {"bytes": size * d * (4 * rows + 4 * keys) + 4 * rows, "flops": 14 * pairs * d}
    return {"bytes": nbytes, "flops": 4 * pairs * filled * d}


def tolerance(case):
    """About four times the distance from a float64 evaluation of the same pass, measured on the listed cases and on
    sixteen smaller drawn ones: bf16 attention 2.3e-3 (largest element 1.8e-2, 3e-2 under the causal mask, whose first
    rows are larger than the rest), gradients 2.5e-3 (1.2e-1), encoder block 2.9e-3 (1.5e-2), fp32 1.0e-6 (9e-6)."""
    if case.get("fp32"):
        return {"rel": 4e-6, "max": 4e-5}
    if case["kind"] == "training":
        return {"rel": 0.01, "max": 0.5}
    if case["kind"] == "block":
        return {"rel": 0.012, "max": 0.06}
    return {"rel": 0.01, "max": 0.12 if case.get("causal") else 0.08}
