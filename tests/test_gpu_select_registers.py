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


@pytest.mark.parametrize("n,lists", [(100, 3), (2500, 3), (9000, 3), (9000, 400), (20000, 3), (40000, 3)])
def test_order_of_special_values(n, lists):
    """-0 is below +0, a NaN without its sign bit is above +inf and one with it below -inf, in every form of both steps; ties, NaNs of
    the same bits among them, go to the lowest index.  Against a stable sort of the 32-bit images."""
    gen = torch.Generator(device=DEV).manual_seed(n)
    v = torch.randn(lists, n, generator=gen, device=DEV)
    kinds = torch.randint(0, 12, (lists, n), generator=gen, device=DEV)
    for k, bits in enumerate((0, -2 ** 31, 0x7f800000, -0x800000, 0x7fc00000, -0x400000, 0x7fc00001, 1)):
        v = torch.where(kinds == k, torch.full_like(kinds, bits).to(torch.int32).view(torch.float32), v)
    image = v.view(torch.int32)
    image = torch.where(image < 0, image ^ 0x7fffffff, image)
    sh = vec.Shape(1, 1, lists, lists, 64, vec.VECTOR_F32, 1)
    for k in (n // 16 * 2, n // 4 * 2, n // 2 * 2 - 2):
        out = torch.empty(lists, k, dtype=torch.int32, device=DEV)
        vec.vector_pool_select(sh, vec.Budget(n, k, 0, k, 0, k, n - k), v, out)
        assert torch.equal(out.long(), torch.sort(image, dim=1, descending=True, stable=True).indices[:, :k].sort(dim=1).values), k
        pool = torch.arange(n, dtype=torch.int32, device=DEV).repeat(lists, 1).contiguous()
        tier = torch.empty(lists, n, dtype=torch.uint8, device=DEV)
        ret, apx = (torch.empty(lists, m, dtype=torch.int32, device=DEV) for m in (n - k, k))
        vec.vector_truncate(sh, vec.Budget(n, n - k // 2, k // 2, n, k, n - k, 0), v, pool, tier, ret, apx)
        order = torch.sort(image, dim=1, stable=True).indices
        assert torch.equal(apx.long(), order[:, :k].sort(dim=1).values) and torch.equal(ret.long(), order[:, k:].sort(dim=1).values), k
