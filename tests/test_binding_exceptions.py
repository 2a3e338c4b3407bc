"""Tensors without memory of their own (those that vmap, grad and tracing hand a function) raise torch's error from every call;
the process lives on.  No GPU needed: the tensors only say that they are on one."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2107_06419_b200 import api

H, N, d, D = 4, 128, 64, 256
def t(*shape, dtype=torch.bfloat16):
    return torch.empty(2, *shape, device="cuda", dtype=dtype)
q = lambda: t(1, H, N, d)
f = lambda: t(1, H, N, dtype=torch.float32)
x = lambda: t(1, N, D)
calls = {
    "fwd": (lambda q, k, v, o: api.flat_attn_fwd(q, k, v, o, 1.0), [q, q, q, q]),
    "fwd_ex": (lambda q, k, v, o, l, n: api.flat_attn_fwd_ex(q, k, v, o, 1.0, lse=l, k_valid_len=n),
               [q, q, q, q, f, lambda: t(1, dtype=torch.int32)]),
    "bwd": (lambda q, k, v, o, g, l, a, b, c, e: api.flat_attn_bwd(q, k, v, o, g, l, a, b, c, e, 1.0), [q] * 5 + [f] + [q] * 3 + [f]),
    "bwd_ex": (lambda q, k, v, o, g, l, a, b, c, e: api.flat_attn_bwd_ex(q, k, v, o, g, l, a, b, c, e, 1.0),
               [q] * 5 + [f] + [q] * 3 + [f]),
    "varlen": (lambda q, k, v, o, a, b: api.flat_attn_varlen_fwd(q, k, v, o, a, b, N, 1.0),
               [lambda: t(N, H, d)] * 4 + [lambda: t(3, dtype=torch.int32)] * 2),
    "layer": (lambda *a: api.flat_attn_layer_fwd(*a, 1.0), [x, lambda: t(3 * D, D), lambda: t(D, D), x] + [q] * 4),
    "fc": (lambda *a: api.flat_fc_fwd(*a), [x, lambda: t(D, D), x]),
    "layernorm": (lambda *a: api.flat_layernorm_fwd(*a), [x, lambda: t(D), lambda: t(D), x]),
    "status": (lambda q, k, v, o, s: api.flat_attn_fwd_ex(q, k, v, o, 1.0, status=s), [q, q, q, q, lambda: t(1, dtype=torch.int32)]),
}
call, make = calls[%r]
with FakeTensorMode():
    try:
        torch.vmap(call)(*(m() for m in make))
    except RuntimeError as e:
        assert "data pointer" in str(e), e
        print("raised")
"""


@pytest.mark.parametrize("name", ["fwd", "fwd_ex", "bwd", "bwd_ex", "varlen", "layer", "fc", "layernorm", "status"])
def test_tensors_without_memory_raise(name):
    r = subprocess.run([sys.executable, "-c", PROGRAM % name], cwd=ROOT, capture_output=True, text=True, env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0 and r.stdout.strip() == "raised", r.stdout + r.stderr[-2000:]


def test_a_stream_that_is_no_address():
    """A whole number too large for an address is handed back like every argument that is not plain, with no error left behind."""
    code = """
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2107_06419_b200 import api
def call(x):
    print(api._binding.fc_fwd(x, x, x, None, 1 << 80))      # (the shapes do not match either: nothing asks for the memory)
    return x
with FakeTensorMode():
    torch.vmap(call)(torch.empty(2, 128, 64, device="cuda", dtype=torch.bfloat16))
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0 and r.stdout.strip() == "-1", r.stdout + r.stderr[-2000:]
