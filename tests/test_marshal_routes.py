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


class _Handle:
    def __init__(self, stream):
        self.cuda_stream = stream.cuda_stream


@pytest.mark.gpu
@pytest.mark.parametrize("form", ["object", "handle", "wrapped", "default"])
def test_a_given_stream(monkeypatch, form):
    """Every call of a loop on a given stream, without ctypes, against ctypes on the same stream; the stream that it says is the one that
    runs it: work queued there ahead of the call is seen by it."""
    sh = vec.Shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16)
    got = []
    for plain in (True, False):
        side = torch.cuda.default_stream() if form == "default" else torch.cuda.Stream()
        st = {"object": side, "handle": side.cuda_stream, "wrapped": _Handle(side), "default": 0}[form]
        c, q, W, k, v = _problem(sh)
        b, ws = c.budget, c.ws
        K, Q = torch.randn(2, N, D, generator=torch.Generator().manual_seed(1)).cuda().bfloat16(), q.repeat_interleave(16, 1).view(2, 2, 16, D).contiguous()
        out, out2 = (torch.zeros(2, 2, D, device="cuda") for _ in range(2))
        k2, big = torch.zeros_like(k), torch.zeros(64 << 20, device="cuda")
        torch.cuda.synchronize()
        with monkeypatch.context() as m:
            if plain:
                _no_ctypes(m)
            else:
                m.setattr(B, "_marshal_module", _Nothing())
            with torch.cuda.stream(side):
                for _ in range(20):
                    big.add_(1)
                k2.copy_(k)
            vec.vector_score(sh, Q, K, N, c.scores, None, ws, st)
            vec.vector_route(sh, b, c.scores, K, K, W, c.tier, c.ret_idx, c.apx_idx, None, None, ws, st)
            c.cache.n_ret = b.n_ret
            vec.vector_compact(sh, b, K, K, c.ret_idx, c.apx_idx, c.cache, st)
            vec.vector_append(sh, c.cache, k2, v, N, st)
            c.cache.n_ret += 1
            vec.vector_decode_attn(sh, q, c.cache, W, out, 0, ws, st)
            vec.vector_decode_attn_static(sh, q, c.cache, W, out2, 0, st)
        torch.cuda.synchronize()
        assert torch.equal(c.cache.ret_k[:, c.cache.n_ret - 1], k)
        got.append((c.scores, c.tier, c.ret_idx, c.apx_idx, c.cache.ret_k[:, :c.cache.n_ret], c.cache.ret_v[:, :c.cache.n_ret], out, out2))
    assert all(torch.equal(a, b) for a, b in zip(*got))


class _Nothing:
    """Leaves every call to ctypes."""

    def __getattr__(self, name):
        return lambda *args: None


class _Shape(vec.Shape):
    """A program's own shape."""


class _Cache(vec.Cache):
    """A program's own cache."""


class _Packs(vec.Shape):
    """One that packs in its own way: the module may not read it."""

    def _p(self):
        return vec.Shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16)._p()


class _Typed(vec.Shape):
    torch_dtype = torch.bfloat16


class _PacksCache(vec.Cache):
    def _p(self):
        return vec.Cache._p(self)


@pytest.mark.gpu
@pytest.mark.parametrize("shape,cache", [(_Shape, vec.Cache), (vec.Shape, _Cache), (_Shape, _Cache), (_Packs, vec.Cache), (_Typed, vec.Cache), (vec.Shape, _PacksCache)])
def test_appending_with_classes_of_the_program(shape, cache):
    """One kernel, as for the binding's own classes; rows that it refuses are assigned."""
    c, q, W, k, v = _problem(vec.Shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16))
    c.shape, o = shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16), c.cache
    c.cache = cache(o.ret_k, o.ret_v, o.apx_k, o.ret_pos, o.apx_pos, o.n_ret, o.n_apx)
    n, before = c.cache.n_ret, vec.vector_kernel_launches()
    c.append(k, v, N)
    assert vec.vector_kernel_launches() == before + 1 and c.cache.n_ret == n + 1
    shifted = torch.empty(2 * D + 1, dtype=torch.bfloat16, device="cuda")[1:].view(2, D).copy_(k)
    for i, (a, b) in enumerate(((k.double(), v), (shifted, v), (k, v[:1]))):
        c.append(a, b, N + 1 + i)
    assert vec.vector_kernel_launches() == before + 1 and c.cache.n_ret == n + 4
    assert all(torch.equal(c.cache.ret_k[:, n + i], k) for i in range(4)) and torch.equal(c.cache.ret_v[:, n + 1], v)
    assert torch.equal(c.cache.ret_pos[:, n:n + 4], torch.arange(N, N + 4, device="cuda", dtype=torch.int32).expand(2, 4))
    with pytest.raises(ValueError):
        c.append(k, v, N)


@pytest.mark.gpu
def test_which_classes_the_module_reads():
    c, q, W, k, v = _problem(vec.Shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16))
    o, out = c.cache, torch.empty(2, 2, D, device="cuda")
    for shape, cache, read in ((vec.Shape, vec.Cache, True), (_Shape, _Cache, True), (_Packs, vec.Cache, False), (_Typed, vec.Cache, False), (vec.Shape, _PacksCache, False)):
        rc = B._marshal().decode_attn(shape(1, 1, 4, 2, D, vec.VECTOR_BF16, 16), q, cache(o.ret_k, o.ret_v, o.apx_k, o.ret_pos, o.apx_pos, o.n_ret, o.n_apx),
                                      W, out, 0, c.ws, None)
        assert rc == 0 if read else rc is None
