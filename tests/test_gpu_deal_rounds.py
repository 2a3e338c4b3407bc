"""Equal items in a few rounds, the last one mostly empty: the key steps dealt evenly, with one, two and three items per SM."""
import numpy as np
import pytest
import torch

import oracle
from paper_2107_06419_b200 import inputs
from helpers import bf16_tensor, bf16_to_f64, check_bf16, rand_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [(1, 20, 2000, 2000), (5, 10, 1500, 1500), (3, 50, 769, 1700), (2, 6, 4930, 4930)], ids=str)
def test_deal_of_equal_items(case):
    from paper_2107_06419_b200 import api
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expected choices are those of a 148-SM GPU")
    B, H, Nq, Nk = case
    rng = np.random.default_rng(Nq)
    Qb, Kb, Vb = rand_bits(rng, (B, H, Nq, 64)), rand_bits(rng, (B, H, Nk, 64)), rand_bits(rng, (B, H, Nk, 64))
    rows = inputs.sample_rows(inputs.Workload("deal", B, H, Nq, Nk, 64), 24)
    ref = oracle.attention(Qb, Kb, Vb, 0.125, rows=rows)["O"]
    Q, K, V = bf16_tensor(Qb), bf16_tensor(Kb), bf16_tensor(Vb)
    first = None
    for _ in range(3):
        O = torch.full(Q.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        api.flat_attn_fwd_ex(Q, K, V, O, 0.125, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and api.flat_attn_last_schedule() == api.FLAT_SCHEDULE_EVEN_DEAL
        check_bf16(bf16_to_f64(O.reshape(-1, 64)[torch.from_numpy(rows).cuda()]), ref, "deal")
        assert first is None or torch.equal(O, first)
        first = O


@pytest.mark.parametrize("B,H,N,dealt", [(3, 12, 1500, True), (1, 26, 2048, True), (1, 30, 1600, True), (1, 40, 1500, False), (1, 17, 4096, False)])
def test_line_of_the_deal(B, H, N, dealt):
    """Less than one and a half items per SM: dealt; above, with few key steps: whole."""
    from paper_2107_06419_b200 import api
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the expected choices are those of a 148-SM GPU")
    torch.manual_seed(N)
    Q, K, V = (torch.randn(B, H, N, 64, device="cuda").to(torch.bfloat16) for _ in range(3))
    O = torch.full_like(Q, float("nan"))
    torch.cuda.synchronize()
    api.flat_attn_fwd(Q, K, V, O, 0.125)
    torch.cuda.synchronize()
    assert api.flat_attn_last_variant() == api.FLAT_VARIANT_TC3
    assert (api.flat_attn_last_schedule() == api.FLAT_SCHEDULE_EVEN_DEAL) == dealt
    ref = torch.softmax(Q.float() @ K.float().transpose(2, 3) * 0.125, -1) @ V.float()
    assert float((O.float() - ref).abs().max()) <= 2e-2  # (the parity bar of bf16 results)
