"""fp32 tensors with head sizes 32 and 128 (split-tf32 products) at the edges of their key steps and query tiles, against the oracle
and against the FFMA kernel; masks, lse, values at the ends of the fp32 range."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def run(api, Q, K, V, scale, variant=0, vl=None, causal=False):
    Qt, Kt, Vt = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (Q, K, V))
    O = torch.full(Qt.shape, float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    lse = torch.full(Qt.shape[:3], float("nan"), device="cuda")
    api.flat_attn_fwd_ex(Qt, Kt, Vt, O, scale, k_valid_len=None if vl is None else torch.from_numpy(vl).cuda(), status=status,
                         variant=variant, causal=causal, lse=lse)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return O.double().cpu().numpy(), lse.double().cpu().numpy()


@pytest.mark.parametrize("d", [32, 128])
@pytest.mark.parametrize("Nk", [1, 31, 32, 33, 63, 64, 65, 96, 128, 129, 333])
def test_edges(d, Nk):
    from paper_2107_06419_b200 import api
    for Nq, causal, vl, scale in ((1, False, None, d ** -0.5), (129, True, None, d ** -0.5), (300, False, [Nk, Nk // 2], -d ** -0.5)):
        rng = np.random.default_rng(Nq + 7 * Nk + d)
        Q, K, V = (rng.standard_normal((2, 3, n, d)).astype(np.float32) for n in (Nq, Nk, Nk))
        vl = None if vl is None else np.array(vl, dtype=np.int32)
        ref = oracle.attention(Q, K, V, scale, valid_len=vl, causal=causal, want_lse=True)
        O, lse = run(api, Q, K, V, scale, vl=vl, causal=causal)
        assert api.flat_attn_last_variant() == api.FLAT_VARIANT_TF32
        F, _ = run(api, Q, K, V, scale, variant=api.FLAT_VARIANT_SIMT, vl=vl, causal=causal)
        live = np.isfinite(ref["LSE"])
        assert np.all(O[~live] == 0.0) and np.all(np.isneginf(lse[~live]))
        # a logit |q . k| scale is off by at most 2^-20 of sum |q k| scale (three products: 2^-22 dropped, 2^-22 for x_lo as a tf32
        # number, and the rounding of d sums), a weight by that much in base e, the output by twice that over the largest |v|
        logit = 2.0 ** -20 * abs(scale) * np.abs(Q).sum(-1).max() * np.abs(K).max()
        bound = 2 * logit * np.abs(V).max() + 2.0 ** -20 * np.abs(V).max()
        assert np.max(np.abs(O - ref["O"])) <= bound
        assert np.max(np.abs(lse[live] - ref["LSE"][live]), initial=0.0) <= logit + 2e-6
        # on the whole no less exact than the FFMA kernel: its error, and one rounding of the operands to 23 bits
        rms = lambda e: float(np.sqrt(np.mean(e * e)))
        assert rms(O - ref["O"]) <= 1.5 * rms(F - ref["O"]) + 2.0 ** -23 * np.abs(V).max() / 4


@pytest.mark.parametrize("d", [32, 128])
def test_ends_of_the_range(d):
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(d)
    Q, K = (rng.standard_normal((1, 1, n, d)).astype(np.float32) for n in (40, 70))
    V = rng.standard_normal((1, 1, 70, d)).astype(np.float32)
    big = np.finfo(np.float32).max
    V[..., 0] = big / 128                                # (70 weights of at most 1 each: no partial sum passes the largest number)
    V[..., 1] = 1e-38
    V[..., 2] = 0.0
    O, _ = run(api, Q, K, V, d ** -0.5)
    ref = oracle.attention(Q, K, V, d ** -0.5)["O"]
    assert np.all(np.isfinite(O)) and np.all(O[..., 2] == 0.0)
    assert np.max(np.abs(O[..., 0] / ref[..., 0] - 1)) <= 1e-5
    assert np.max(np.abs(O[..., 1] - ref[..., 1])) <= 2.0 ** -10 * 1e-38 + 1e-44
    assert np.max(np.abs(O[..., 3:] - ref[..., 3:])) <= 2e-5
    # one visible key: its values, the largest number of either sign included, whose head must not be rounded to infinity
    V[..., 0], V[..., 3] = big, -big
    one, _ = run(api, Q, K, V, d ** -0.5, vl=np.array([1], dtype=np.int32))
    assert np.all(np.isfinite(one)) and np.max(np.abs(one[..., [0, 3]] / V[0, 0, 0, [0, 3]].astype(np.float64) - 1)) <= 2.0 ** -20


@pytest.mark.parametrize("d", [32, 64, 128])
def test_odd_number_of_key_steps(d):
    """The stream of the odd key steps ends before the last even one: many times over, the same results."""
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(d)
    Nk = 5 * (32 if d == 128 else 64) - 40
    Q, K, V = (rng.standard_normal((6, 12, n, d)).astype(np.float32) for n in (300, Nk, Nk))
    ref = oracle.attention(Q, K, V, d ** -0.5)["O"]
    first = None
    for _ in range(10):
        O, _ = run(api, Q, K, V, d ** -0.5)
        assert np.max(np.abs(O - ref)) <= 2e-5
        assert first is None or np.array_equal(O, first)
        first = O


@pytest.mark.parametrize("heads,Nq,Nk,simt", [(16, 64, 64, False), (1024, 64, 64, True), (1024, 1, 16, True), (1024, 64, 65, False),
                                              (1024, 65, 64, False)])
def test_many_heads_of_one_tile(heads, Nq, Nk, simt):
    """d = 32: one FFMA tile a head and more heads than SMs run on the FFMA kernel."""
    from paper_2107_06419_b200 import api
    rng = np.random.default_rng(heads + Nq + Nk)
    Q, K, V = (rng.standard_normal((1, heads, n, 32)).astype(np.float32) for n in (Nq, Nk, Nk))
    O, lse = run(api, Q, K, V, 32 ** -0.5)
    assert api.flat_attn_last_variant() == (api.FLAT_VARIANT_SIMT if simt else api.FLAT_VARIANT_TF32)
    ref = oracle.attention(Q, K, V, 32 ** -0.5, want_lse=True)
    assert np.max(np.abs(O - ref["O"])) <= 2e-5 and np.max(np.abs(lse - ref["LSE"])) <= 2e-5
