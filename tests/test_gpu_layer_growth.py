"""Decode with a layer's map where the running maximum moves along the tokens: by little at a time, which leaves the
softmax's reference behind, and by jumps, which move it; ragged ends of both pools, one pool alone, fewer tiles than
stages; and where a block's share of the tiles begins and ends inside a (sequence, layer) pair.  Tolerance: 2e-2
absolute, as for the layer-map decode elsewhere."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("L,B,g,n_ret,n_apx,jump", [
    (10, 10, 4, 100, 700, 0.0),                  # fewer pairs than multiprocessors, blocks across their ends
    (40, 4, 1, 17, 33, 0.0),                     # more pairs than multiprocessors, four tiles each
    (19, 8, 2, 0, 130, 20.0),
    (3, 1, 4, 1600, 3300, 0.0),                  # 49 blocks' worth a pair: the limit of records
])
def test_decode_layer_pieces(oracle, L, B, g, n_ret, n_apx, jump):
    _check(oracle, L, B, g, n_ret, n_apx, jump)


@pytest.mark.parametrize("g,n_ret,n_apx,jump", [
    (4, 16 * 20 + 1, 32 * 24 + 31, 0.0),     # logits rise steadily
    (4, 16 * 20 + 15, 32 * 24 + 1, 40.0),    # ... and by a jump in either pool
    (1, 0, 700, 20.0),                       # key-only tokens alone
    (3, 333, 0, 20.0),                       # retained tokens alone
    (2, 5, 0, 0.0),                          # one tile
    (4, 17, 33, 0.0),                        # four tiles
])
def test_decode_layer_growth(oracle, g, n_ret, n_apx, jump):
    _check(oracle, 2, 2, g, n_ret, n_apx, jump)


def _check(oracle, L, B, g, n_ret, n_apx, jump):
    Hkv, d = 8, 128
    UL, U = L * B, L * B * Hkv
    gen = torch.Generator(device=DEV).manual_seed(n_ret + n_apx)
    q = torch.randn(U, g, d, generator=gen, device=DEV)
    q = (q / q.norm(dim=2, keepdim=True) * np.sqrt(d)).to(torch.bfloat16)

    def keys(n):
        """Keys whose logits against the unit's first head grow by about 30 (powers of e) over the pool."""
        k = torch.randn(U, n + 3, d, generator=gen, device=DEV)
        rise = torch.linspace(-10.0, 20.0, n + 3, device=DEV) + jump * (torch.arange(n + 3, device=DEV) > 0.6 * n)
        return (k + rise.view(1, -1, 1) * q[:, :1].float() / np.sqrt(d)).to(torch.bfloat16)
    rk, ak = keys(n_ret), keys(n_apx)
    rv = torch.randn(U, n_ret + 3, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(L, Hkv * d, Hkv * d, generator=gen, device=DEV) / np.sqrt(Hkv * d) * 0.3).to(torch.bfloat16)
    pos = [torch.zeros(U, n + 3, dtype=torch.int32, device=DEV) for n in (n_ret, n_apx)]
    cache = vec.Cache(rk, rv, ak, pos[0], pos[1], n_ret, n_apx)
    sh = vec.Shape(B, L, Hkv * g, Hkv, d, vec.VECTOR_BF16, 16, 7, 0.0, 0, 10000.0)
    ws = torch.empty(vec.vector_layer_workspace_bytes(sh, vec.vector_plan_budget(8192, 4096, -1, 16)), dtype=torch.uint8, device=DEV)
    out = torch.full((U, g, d), float("nan"), dtype=torch.float32, device=DEV)
    vec.vector_decode_attn_layer(sh, q, cache, W, out, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    for ul in sorted({*range(0, UL, max(1, UL // 5)), UL - 1}):
        sl = slice(ul * Hkv, (ul + 1) * Hkv)
        _, o = oracle.attend_layer(q[sl].reshape(Hkv * g, d).cpu(), rk[sl, :n_ret].cpu(), rv[sl, :n_ret].cpu(), ak[sl, :n_apx].cpu(),
                                   W[ul % L].cpu(), 1.0 / np.sqrt(d))
        assert np.max(np.abs(out[sl].reshape(Hkv * g, d).cpu().double().numpy() - o)) <= 2e-2, ul
