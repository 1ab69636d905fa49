"""Selections at the sizes where the number of registers and the number of warps change, and where a warp's piece is empty or ends
inside a register's run of 32: exact (indices and tiers are whole numbers)."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"
SIZES = [1, 31, 33, 511, 513, 2047, 2048, 2049, 4096, 4097, 8192, 8193, 16384, 16385, 20011, 32767, 32768, 32769]


def _values(U, n, kind, seed):
    v = torch.randn(U, n, generator=torch.Generator().manual_seed(seed))
    if kind == "ties":
        v = torch.round(v * 4) / 4 + 0.0
    elif kind == "equal":
        v = torch.full_like(v, 3.0)
    v[:, n // 2] = float("inf")
    v[0, : n // 3] = torch.finfo(torch.float32).min
    return v


@pytest.mark.parametrize("kind", ["random", "ties", "equal"])
@pytest.mark.parametrize("n", SIZES)
def test_selections(oracle, n, kind):
    U = 3
    sh = vec.Shape(1, 1, U, U, 64, vec.VECTOR_F32, 1)
    v = _values(U, n, kind, n)
    for k in sorted({1, (n + 2) // 3, n}):
        out = torch.empty(U, k, dtype=torch.int32, device=DEV)
        vec.vector_pool_select(sh, vec.Budget(n, k, 0, k, 0, k, n - k), v.to(DEV), out)
        for u in range(U):
            assert np.array_equal(out[u].cpu().numpy(), oracle.pool_select(v[u].numpy(), k)), (k, u)
    N = n + 100
    pool = torch.stack([torch.randperm(N, generator=torch.Generator().manual_seed(u))[:n].sort().values for u in range(U)]).to(torch.int32)
    for k in sorted({0, n // 3 // 2 * 2, n // 2 * 2}):
        tier = torch.empty(U, N, dtype=torch.uint8, device=DEV)
        ret, apx = (torch.empty(U, max(m, 1), dtype=torch.int32, device=DEV) for m in (n - k, k))
        vec.vector_truncate(sh, vec.Budget(N, n - k // 2, k // 2, n, k, n - k, N - n), v.to(DEV), pool.to(DEV), tier, ret, apx)
        for u in range(U):
            t, r, a = oracle.truncate(v[u].numpy(), pool[u].numpy(), k, N)
            assert np.array_equal(tier[u].cpu().numpy(), t), (k, u)
            # the lists lie back to back
            assert np.array_equal(ret.flatten()[u * (n - k):(u + 1) * (n - k)].cpu().numpy(), r), (k, u)
            assert np.array_equal(apx.flatten()[u * k:(u + 1) * k].cpu().numpy(), a), (k, u)
