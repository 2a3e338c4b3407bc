"""The backward kernels where their branches change: rows that are switched off, scales at which -lse / scale is extreme, rings
that wrap, and the order of the tiles under the causal mask (bars of tests/test_gpu_bwd.py)."""
import numpy as np
import pytest

import oracle
from helpers import rand_bits
from test_gpu_bwd import api, check_grad, run_fwd_bwd  # noqa: F401  (the fixture and the bars)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("Nq,Nk,causal,scale", [
    (1, 1, False, 0.1), (127, 65, False, 0.1), (129, 128, True, 0.1),
    (700, 900, True, 0.1),                               # six / eight streamed steps: every ring wraps
    (400, 130, True, 0.1),                               # the first 270 queries see no key
    (200, 300, False, -0.1),                             # negative scale: the sign of a switched-off query's term follows it
    (200, 300, True, 0.0), (200, 300, False, 1e-12)])    # lse / scale beyond any logit
def test_backward_edges(api, d, Nq, Nk, causal, scale):  # noqa: F811
    B, H = 2, 3
    rng = np.random.default_rng(Nq + Nk + d)
    Qb, Kb, Vb, dOb = (rand_bits(rng, (B, H, n, d)) for n in (Nq, Nk, Nk, Nq))
    O, lse, dQ, dK, dV = run_fwd_bwd(api, Qb, Kb, Vb, dOb, scale, causal=causal)
    ref = oracle.attention_bwd(Qb, Kb, Vb, dOb, scale, causal=causal)
    for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
        if Nk == 1 and name != "dV":
            # one key: p = 1 and O = V, so dS = dP - delta is the difference of two fp32 sums of the same d products (each
            # of order 1): 2 d sums of relative error 2^-24, at most 1e-4 together
            assert np.abs(got).max() <= 1e-4, name
        elif np.abs(ref[name]).max() == 0:
            assert np.all(got == 0), name
        else:
            check_grad(got, ref[name], "%s %s" % (name, (Nq, Nk, causal, scale)))
