"""Decode with one map per layer, merged for several sequences a block: batches that divide among the blocks and ones that do not,
and numbers of query heads that leave columns of the product empty.  Against the oracle, element-wise: two per cent of one, the
tolerance that every decode test has (outputs are of size one; another sequence's or head's output is off by that much).  Outputs in
bf16 are the fp32 ones rounded."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("batch,layers,g,n_ret,n_apx", [(5, 8, 4, 40, 70), (9, 8, 1, 33, 64), (7, 9, 2, 100, 30), (20, 2, 3, 17, 200), (21, 2, 3, 20, 90),
                                                      (2, 30, 4, 16, 0), (3, 1, 4, 0, 500)])      # the last: few units, a sequence a block
def test_batches(oracle, batch, layers, g, n_ret, n_apx):
    H, d = 8, 128
    U = batch * layers * H
    assert batch == 3 or U > 2 * torch.cuda.get_device_properties(0).multi_processor_count      # where blocks share the map
    gen = torch.Generator(device=DEV).manual_seed(batch * 100 + g)
    sh = vec.Shape(batch, layers, H * g, H, d, vec.VECTOR_BF16, 16)
    rand = lambda *s: torch.randn(*s, generator=gen, device=DEV).to(torch.bfloat16)
    n_pool, n_a = n_ret + n_apx, n_apx // 2
    budget = vec.Budget(4 * n_pool, n_pool - n_a, n_a, n_pool, n_apx, n_ret, 3 * n_pool)
    cache = vec.Cache(rand(U, max(n_ret, 1), d), rand(U, max(n_ret, 1), d), rand(U, max(n_apx, 1), d),
                      torch.zeros(U, max(n_ret, 1), dtype=torch.int32, device=DEV), torch.zeros(U, max(n_apx, 1), dtype=torch.int32, device=DEV), n_ret, n_apx)
    W = (torch.randn(layers, H * d, H * d, generator=gen, device=DEV) / np.sqrt(H * d)).to(torch.bfloat16)
    q = rand(U, g, d)
    out = torch.full((U, g, d), float("nan"), device=DEV)
    ws = torch.empty(vec.vector_layer_workspace_bytes(sh, budget), dtype=torch.uint8, device=DEV)
    vec.vector_decode_attn_layer(sh, q, cache, W, out, ws)
    out16 = torch.full((U, g, d), float("nan"), device=DEV, dtype=torch.bfloat16)
    vec.vector_decode_attn_layer(sh, q, cache, W, out16, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    assert torch.equal(out16, out.to(torch.bfloat16))
    for ul in sorted({0, layers, (batch // 2) * layers + layers - 1, batch * layers - 1} & set(range(batch * layers))):
        sl = slice(ul * H, (ul + 1) * H)
        _, want = oracle.attend_layer(q[sl].reshape(H * g, d).cpu(), cache.ret_k[sl, :n_ret].cpu(), cache.ret_v[sl, :n_ret].cpu(),
                                      cache.apx_k[sl, :n_apx].cpu(), W[ul % layers].cpu(), d ** -0.5)
        assert np.max(np.abs(out[sl].reshape(H * g, d).cpu().double().numpy() - want)) <= 2e-2, ul
