"""The extension module that marshals arguments: the plain case gives what ctypes gives, anything else is left to ctypes, which refuses
what it refused."""
import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import binding as B
from paper_2605_23258_b200.pipeline import Compressor


class _Sub(vec.Shape):
    pass


def test_anything_but_the_plain_case_is_left_to_ctypes():
    m = B._marshal()
    sh, budget = vec.Shape(1, 1, 4, 2, 64, vec.VECTOR_F32, 16), vec.vector_plan_budget(200, 60, 10, 16)
    q, k, s = torch.zeros(2, 2, 16, 64), torch.zeros(2, 200, 64), torch.zeros(2, 200)
    assert m.score(sh, q, k, 200, s, None, None, None) is None                      # host memory
    for bad in (_Sub(1, 1, 4, 2, 64, vec.VECTOR_F32, 16), vec.Shape(1, 1, 4, 2, 64, vec.VECTOR_F32, 16.0), vec.Shape(1, 1, 2**31, 2, 64, vec.VECTOR_F32, 16),
                vec.Shape(1, 1, 4, 2, 64, vec.VECTOR_F32, 16, 7, 0), None):
        assert m.score(bad, None, None, 200, None, None, None, 0) is None
    assert m.score(sh, None, None, 2**70, None, None, None, None) is None
    assert m.score(sh, torch.nn.Module, None, 200, None, None, None, None) is None
    assert m.route(sh, None, *[None] * 11) is None and m.append_rows(sh, None, q, q, 0) is None
    with pytest.raises(TypeError):
        m.score(sh)
    for name, args in (("vector_score", (sh, q, k, 200, s)), ("vector_route", (sh, budget, s, k, k, k, s, s, s)),
                       ("vector_decode_attn", (sh, q, Compressor(sh, budget, device="cpu").cache, k, s))):
        with pytest.raises(ValueError, match="must be a CUDA tensor"):
            getattr(vec, name)(*args)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_plain_calls_give_what_ctypes_gives(dtype):
    """Every call by either route, ctypes by way of an explicit stream; and each refusal."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.randn(*s, generator=gen, device="cuda").to(dtype)
    N, d, H, g, w = 700, 64, 2, 2, 16
    sh = vec.Shape(1, 2, H * g, H, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, w)
    U, budget, stream = sh.units, vec.vector_plan_budget(N, N // 4, -1, w), torch.cuda.current_stream()
    K, V, Q, W, WL, q = rand(U, N, d), rand(U, N, d), rand(U, g, w, d), rand(U, d, d) / 8, rand(2, H * d, H * d) / 12, rand(U, g, d)
    kn, vn = rand(U, d), rand(U, d)
    m = B._marshal()
    got = []
    for st in (None, stream):
        c = Compressor(sh, budget, extra_rows=2)
        for t in (c.cache.ret_k, c.cache.ret_v, c.cache.apx_k, c.cache.ret_pos, c.cache.apx_pos):
            t.zero_()
        ws = torch.empty(max(c.ws.numel(), vec.vector_layer_workspace_bytes(sh, budget)), dtype=torch.uint8, device="cuda")
        raw, out, out2 = torch.empty(U, N, device="cuda"), torch.empty(U, g, d, device="cuda"), torch.empty(U, g, d, dtype=torch.bfloat16, device="cuda")
        vec.vector_score(sh, Q, K, N, c.scores, raw, ws, st)
        vec.vector_route(sh, budget, c.scores, K, V, W, c.tier, c.ret_idx, c.apx_idx, None, None, ws, st)
        vec.vector_compact(sh, budget, K, V, c.ret_idx, c.apx_idx, c.cache, st)
        if st is None:
            assert B.append_rows(sh, c.cache, kn, vn, N)
        else:
            vec.vector_append(sh, c.cache, kn, vn, N, st)
        c.cache.n_ret += 1
        vec.vector_decode_attn(sh, q, c.cache, W, out, 0, ws, st)
        vec.vector_decode_attn_static(sh, q, c.cache, W, out2, 0, st)
        tier, ret, apx = torch.empty(2, N, dtype=torch.uint8, device="cuda"), c.ret_idx[:2].clone(), c.apx_idx[:2].clone()
        vec.vector_route_layer(sh, budget, c.scores[:2].contiguous(), K, V, WL, tier, ret, apx, None, None, ws, st)
        one = [t.clone() for t in (c.tier, c.ret_idx, c.apx_idx, c.cache.ret_k, c.cache.ret_v, c.cache.apx_k, c.cache.ret_pos, c.cache.apx_pos)]
        c.cache.n_ret = budget.n_ret
        vec.vector_compact_layer(sh, budget, K, V, ret, apx, c.cache, st)
        outl = torch.empty(U, g, d, device="cuda")
        vec.vector_decode_attn_layer(sh, q, c.cache, WL, outl, ws, st)
        got.append([c.scores, raw, *one, out, out2, tier, ret, apx, c.cache.ret_k, c.cache.ret_v, c.cache.apx_k, outl])
    torch.cuda.synchronize()
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert m.score(sh, Q, K, N, c.scores, None, ws, None) == 0 and m.score(sh, Q, K, N, c.scores, None, ws, stream) is None
    assert m.score(sh, Q, K, 1, c.scores, None, ws, None) == -2                      # the library's own refusals come back as they are
    for args in ((sh, Q.double(), K, N, c.scores), (sh, Q, K.transpose(1, 2), N, c.scores), (sh, Q, K, N, c.scores.cpu())):
        with pytest.raises(ValueError):
            vec.vector_score(*args, None, ws)
    with pytest.raises(vec.VectorError) as e:
        vec.vector_score(sh, Q, K, N, c.scores, None, ws[:16])
    assert e.value.status == -5
    full = c.cache.ret_k.shape[1]
    assert not B.append_rows(sh, vec.Cache(c.cache.ret_k, c.cache.ret_v, c.cache.apx_k, c.cache.ret_pos, c.cache.apx_pos, full, 0), kn, vn, 0)
    assert not B.append_rows(sh, c.cache, kn.requires_grad_(), vn, 0) and not B.append_rows(sh, c.cache, vn, vn[:, :32], 0)
