"""Streaming decode under RoPE decoupling against the oracle, more units than the one-launch form takes: key-only tiles that
end in their first or second half, units that begin and end inside a block, teams that meet no key-only tile or no tile at
all, one to eight heads.  Tolerance: 2e-2 absolute, as for the form without rotation; turned keys carry eleven bits."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("U,g,n_ret,n_apx", [
    (75, 1, 1, 1),                 # two tiles a unit, one row each
    (80, 8, 70, 1000),             # eight key-only tiles, the last of 104 rows
    (150, 4, 300, 0),              # retained tiles alone
    (90, 3, 0, 321),               # key-only tiles alone, the last of 65 rows: one row in its second half
    (76, 5, 640, 6400),            # buffers and slots used over and over
])
def test_decode_stream_rope(oracle, d, U, g, n_ret, n_apx):
    gen = torch.Generator(device=DEV).manual_seed(U * 10 + g)
    rk, rv = (torch.randn(U, n_ret + 2, d, generator=gen, device=DEV).to(torch.bfloat16) for _ in range(2))
    ak = torch.randn(U, n_apx + 1, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / np.sqrt(d)).to(torch.bfloat16)
    q = (torch.randn(U, g, d, generator=gen, device=DEV) * 2).to(torch.bfloat16)
    pos = torch.randint(0, 131072, (U, n_apx + 1), generator=gen, device=DEV, dtype=torch.int32)
    cache = vec.Cache(rk, rv, ak, torch.zeros(U, n_ret + 2, dtype=torch.int32, device=DEV), pos, n_ret, n_apx)
    sh = vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16, 16, 7, 0.0, 1, 10000.0)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16))
    out = torch.full((U, g, d), float("nan"), dtype=torch.float32, device=DEV)
    for _ in range(2):             # the second call meets the records of the first
        vec.vector_decode_attn(sh, q, cache, W, out, 0, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    for u in sorted({0, 1, U // 2, U - 2, U - 1}):
        _, o = oracle.attend(q[u].cpu(), rk[u, :n_ret].cpu(), rv[u, :n_ret].cpu(), ak[u, :n_apx].cpu(), W[u].cpu(),
                             1.0 / np.sqrt(d), apx_pos=pos[u, :n_apx].cpu().numpy(), rope=True, theta=10000.0)
        assert np.max(np.abs(out[u].cpu().double().numpy() - o)) <= 2e-2, u
