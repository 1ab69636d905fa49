"""Rows off a 16-byte boundary, where fp32 calls and 64-channel bf16 calls take them: contiguous views one element into their
storage.  fp32 runs the same kernel with other loads: the same bits.  bf16 changes from the tensor-core kernels to CUDA cores, which
keep fp32's precision as those do: equal to a few times what either is off by (3e-7, a tenth of the bound)."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _shifted(x):
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    y.copy_(x)
    assert y.is_contiguous() and y.data_ptr() % 16
    return y


def _same(got, want, exact):
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    fin = torch.isfinite(want)
    assert torch.equal(fin, torch.isfinite(got))
    if exact:
        assert torch.equal(got, want)
    else:
        assert ((got - want)[fin].double().norm() / want[fin].double().norm()).item() <= 3e-6


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("layers,N,raw", [(1, 2049, False), (20, 1300, True)])
def test_score(dtype, d, layers, N, raw):
    U, g, w = 2 * layers, 3, 50
    gen = torch.Generator(device=DEV).manual_seed(1)
    Q, K = torch.randn(U, g, w, d, generator=gen, device=DEV).to(dtype), torch.randn(U, N, d, generator=gen, device=DEV).to(dtype)
    sh = vec.Shape(1, layers, 2 * g, 2, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, w)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(N, N, 0, w))
    got, want = ([torch.full((U, N), float("nan"), device=DEV) for _ in range(2)] for _ in range(2))
    vec.vector_score(sh, Q, K, N, want[0], want[1] if raw else None, ws)
    vec.vector_score(sh, _shifted(Q), _shifted(K), N, got[0], got[1] if raw else None, ws)
    _same(got[0], want[0], dtype == torch.float32)
    if raw:
        _same(got[1], want[1], dtype == torch.float32)


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("U,n_idx", [(3, 17), (40, 129)])
def test_residual(dtype, d, rope, U, n_idx):
    gen = torch.Generator(device=DEV).manual_seed(2)
    K, V = (torch.randn(U, 300, d, generator=gen, device=DEV).to(dtype) for _ in range(2))
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / np.sqrt(d)).to(dtype)
    idx = torch.stack([torch.randperm(300, generator=gen, device=DEV)[:n_idx].sort().values for _ in range(U)]).to(torch.int32)
    sh = vec.Shape(1, 1, U, U, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, 16, 7, 0.0, int(rope), 10000.0)
    got, want = (torch.full((U, n_idx), float("nan"), device=DEV) for _ in range(2))
    vec.vector_residual(sh, K, V, W, 300, idx, n_idx, want)
    vec.vector_residual(sh, _shifted(K), _shifted(V), _shifted(W), 300, idx, n_idx, got)
    _same(got, want, dtype == torch.float32)


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("U,g,n_ret,n_apx", [(3, 2, 33, 32), (80, 5, 70, 140), (1, 8, 0, 700)])
def test_decode(dtype, d, rope, U, g, n_ret, n_apx):
    gen = torch.Generator(device=DEV).manual_seed(3)
    rk, rv = (torch.randn(U, n_ret + 1, d, generator=gen, device=DEV).to(dtype) for _ in range(2))
    ak = torch.randn(U, n_apx + 1, d, generator=gen, device=DEV).to(dtype)
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / np.sqrt(d)).to(dtype)
    q = torch.randn(U, g, d, generator=gen, device=DEV).to(dtype)
    pos = torch.randint(0, 131072, (U, n_apx + 1), generator=gen, device=DEV, dtype=torch.int32)
    ret_pos = torch.zeros(U, n_ret + 1, dtype=torch.int32, device=DEV)
    sh = vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, 16, 7, 0.0, int(rope), 10000.0)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16))
    got, want = (torch.full((U, g, d), float("nan"), device=DEV) for _ in range(2))
    vec.vector_decode_attn(sh, q, vec.Cache(rk, rv, ak, ret_pos, pos, n_ret, n_apx), W, want, 0, ws)
    vec.vector_decode_attn(sh, _shifted(q), vec.Cache(_shifted(rk), _shifted(rv), _shifted(ak), ret_pos, pos, n_ret, n_apx), _shifted(W), got, 0, ws)
    _same(got, want, dtype == torch.float32)


@pytest.mark.parametrize("n", [500, 9000, 17000])
def test_tier_map(n):
    """A tier map one byte into its storage, in every form of Step 3 (three lists of 9000 are held in registers, 400 are not)."""
    for U in (3, 400):
        gen = torch.Generator(device=DEV).manual_seed(n)
        eps = torch.rand(U, n, generator=gen, device=DEV)
        N, k = (n + 31) // 16 * 16, n // 4 * 2
        pool = torch.arange(N - n, N, dtype=torch.int32, device=DEV).repeat(U, 1).contiguous()
        sh = vec.Shape(1, 1, U, U, 64, vec.VECTOR_F32, 1)
        ret, apx = (torch.empty(U, m, dtype=torch.int32, device=DEV) for m in (n - k, k))
        tiers = torch.full((U, N), 9, dtype=torch.uint8, device=DEV), torch.full((U * N + 1,), 9, dtype=torch.uint8, device=DEV)
        for t in (tiers[0], tiers[1][1:].view(U, N)):
            vec.vector_truncate(sh, vec.Budget(N, n - k // 2, k // 2, n, k, n - k, N - n), eps, pool, t, ret, apx)
        torch.cuda.synchronize()
        assert torch.equal(tiers[0], tiers[1][1:].view(U, N)) and tiers[1][0] == 9
        assert torch.equal(tiers[0].sum(1), torch.full((U,), 2 * (n - k) + k, device=DEV))
