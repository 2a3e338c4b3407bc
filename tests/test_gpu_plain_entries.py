"""The entry points that take their arguments one by one (flat_attn_fwd, flat_attn_bwd) against those that take a parameter block:
called as C functions and through the binding, bit for bit the same."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_plain_and_ex_entries_agree(monkeypatch):
    from paper_2107_06419_b200 import api
    torch.manual_seed(5)
    B, H, Nq, Nk, d, scale = 2, 3, 150, 210, 64, 0.125
    bf = lambda *s: torch.randn(*s, device="cuda").to(torch.bfloat16)
    Q, K, V, dO = bf(B, H, Nq, d), bf(B, H, Nk, d), bf(B, H, Nk, d), bf(B, H, Nq, d)
    lse = torch.empty(B, H, Nq, device="cuda")
    O = torch.empty_like(Q)
    stream = torch.cuda.current_stream().cuda_stream
    at = lambda *ts: [t.data_ptr() for t in ts]

    def forward(how):
        out = torch.full_like(Q, float("nan"))
        how(out)
        torch.cuda.synchronize()
        return out

    def backward(how):
        g = [torch.full_like(t, float("nan")) for t in (Q, K, V)]
        how(*g, torch.full_like(lse, float("nan")))
        torch.cuda.synchronize()
        return g

    api.flat_attn_fwd_ex(Q, K, V, O, scale, lse=lse)
    f_ex = forward(lambda o: api.flat_attn_fwd_ex(Q, K, V, o, scale))
    b_ex = backward(lambda a, b, c, e: api.flat_attn_bwd_ex(Q, K, V, O, dO, lse, a, b, c, e, scale))
    f_c = forward(lambda o: api._check(api._lib.flat_attn_fwd(*at(Q, K, V, o), B, H, Nq, Nk, d, scale, stream)))
    b_c = backward(lambda *g: api._check(api._lib.flat_attn_bwd(*at(Q, K, V, O, dO, lse, *g), B, H, Nq, Nk, d, scale, stream)))
    # the binding must reach the C function of the same name, not the other one
    monkeypatch.setattr(api._binding, "fwd_ex", None)
    monkeypatch.setattr(api._binding, "bwd_ex", None)
    f = forward(lambda o: api.flat_attn_fwd(Q, K, V, o, scale))
    b = backward(lambda *g: api.flat_attn_bwd(Q, K, V, O, dO, lse, *g, scale))
    assert torch.equal(f, f_ex) and torch.equal(f_c, f_ex) and torch.isfinite(f).all()
    for x, y, z in zip(b, b_c, b_ex):
        assert torch.equal(x, z) and torch.equal(y, z) and torch.isfinite(z.float()).all()
