"""Decode of few units in one launch (a thread block cluster per unit) against the oracle: cluster sizes from two to
sixteen, more blocks than heads and the other way round, blocks whose warps get no tile, and the neighbouring sizes that
take the two-kernel form.  Tolerance: 2e-2 absolute, as for the two-kernel form; a bf16 output adds 2^-8 of the value."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("d,U,g,n_ret,n_apx", [
    (128, 1, 8, 65, 0),            # two tiles: a cluster of two, each with one tile
    (128, 3, 1, 700, 1100),        # more blocks than heads
    (128, 17, 8, 129, 300),        # five tiles
    (128, 37, 4, 500, 900),        # clusters of a few blocks
    (128, 74, 3, 100, 200),        # four tiles, at most two blocks a unit
    (128, 75, 2, 100, 200),        # one unit more than that
    (64, 5, 6, 1000, 2500),
    (64, 2, 2, 0, 129),            # key-only tiles alone
])
def test_decode_cluster(oracle, rope, d, U, g, n_ret, n_apx):
    gen = torch.Generator(device=DEV).manual_seed(U * 100 + g)
    rk, rv = (torch.randn(U, n_ret + 2, d, generator=gen, device=DEV).to(torch.bfloat16) for _ in range(2))
    ak = torch.randn(U, n_apx + 1, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / np.sqrt(d)).to(torch.bfloat16)
    q = (torch.randn(U, g, d, generator=gen, device=DEV) * 2).to(torch.bfloat16)
    pos = torch.randint(0, 131072, (U, n_apx + 1), generator=gen, device=DEV, dtype=torch.int32)
    cache = vec.Cache(rk, rv, ak, torch.zeros(U, n_ret + 2, dtype=torch.int32, device=DEV), pos, n_ret, n_apx)
    sh = vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16, 16, 7, 0.0, int(rope), 10000.0)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16))
    outs = [torch.full((U, g, d), float("nan"), dtype=dt, device=DEV) for dt in (torch.float32, torch.bfloat16)]
    for out in outs:
        vec.vector_decode_attn(sh, q, cache, W, out, 0, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    for u in range(0, U, max(1, U // 4)):
        _, o = oracle.attend(q[u].cpu(), rk[u, :n_ret].cpu(), rv[u, :n_ret].cpu(), ak[u, :n_apx].cpu(), W[u].cpu(),
                             1.0 / np.sqrt(d), apx_pos=pos[u, :n_apx].cpu().numpy(), rope=rope, theta=10000.0)
        assert np.max(np.abs(outs[0][u].cpu().double().numpy() - o)) <= 2e-2, u
        assert np.all(np.abs(outs[1][u].cpu().double().numpy() - o) <= 2e-2 + 2.0 ** -8 * np.abs(o)), u
