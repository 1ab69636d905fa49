"""Which calls the extension module takes, and that a call it leaves to ctypes still does what it did: the kernels that a call launches and its
results, with numbers, classes and streams as programs pass them."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import binding as B
from paper_2605_23258_b200.pipeline import Compressor

N, D = 700, 64


def _problem(shape, extra_rows=4):
    gen = torch.Generator(device="cuda").manual_seed(11)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    U, g, w = int(shape.units), int(shape.group), int(shape.window)
    c = Compressor(shape, vec.vector_plan_budget(N, N // 4, -1, w), extra_rows=extra_rows)
    K, V, Q, W, q = rand(U, N, D), rand(U, N, D), rand(U, g, w, D), rand(U, D, D) / 8, rand(U, g, D)
    c.compress(Q, K, V, W)
    return c, q, W, rand(U, D), rand(U, D)


def _no_ctypes(monkeypatch):
    def refuse():
        raise AssertionError("the call went through ctypes")
    B._marshal()
    monkeypatch.setattr(B, "load_library", refuse)


@pytest.mark.gpu
@pytest.mark.parametrize("fields", [dict(rope_theta=500000), dict(sm_scale=1), dict(batch=np.int64(1), window=np.int32(16)), dict(rope_theta=np.float32(1e6)), dict(rope_enabled=True)])
def test_numbers_as_configurations_hold_them(monkeypatch, fields):
    """A whole step without ctypes, the same as with fields of exactly the declared types."""
    plain = {k: float(v) if k in ("rope_theta", "sm_scale") else int(v) for k, v in fields.items()}
    got = []
    for f in (plain, fields):
        sh = vec.Shape(**{**dict(batch=1, n_layers=1, n_q_heads=4, n_kv_heads=2, head_dim=D, dtype=vec.VECTOR_BF16, window=16), **f})
        c, q, W, k, v = _problem(sh)
        out, before = torch.empty(2, 2, D, device="cuda"), vec.vector_kernel_launches()
        with monkeypatch.context() as m:
            _no_ctypes(m)
            c.append(k, v, N)
            c.cache.n_ret = np.int64(c.cache.n_ret)
            c.append(v, k, N + 1)
            c.decode(q, W, out)
        torch.cuda.synchronize()
        assert vec.vector_kernel_launches() == before + 3
        got.append((out, c.cache.ret_k[:, :c.cache.n_ret], c.cache.ret_pos[:, :c.cache.n_ret]))
    assert all(torch.equal(a, b) for a, b in zip(*got))


def test_numbers_that_are_refused():
    """What struct.pack refuses, the module leaves to it."""
    sh = dict(batch=1, n_layers=1, n_q_heads=4, n_kv_heads=2, head_dim=D, dtype=vec.VECTOR_BF16, window=16)
    budget = vec.vector_plan_budget(200, 60, 10, 16)
    t = torch.zeros(2, D)
    for bad in (dict(window=16.0), dict(batch=2**31), dict(rope_theta="1e4"), dict(sm_scale=2**2000), dict(head_dim=None)):
        assert B._marshal().decode_attn(vec.Shape(**{**sh, **bad}), t, Compressor(vec.Shape(**sh), budget, device="cpu").cache, t, t, 0, None, None) is None
        with pytest.raises(Exception) as e:
            vec.vector_workspace_bytes(vec.Shape(**{**sh, **bad}), budget)
        assert type(e.value).__module__ in ("struct", "builtins")
