"""Residuals with one map per layer on the tensor-core kernel: odd numbers of heads, list ends around a tile, so few tiles that
each is cut in two, and so many that blocks' ranges end inside tiles.  Bound: fp32 accumulation of exact products over
Hkv d inputs in any order, |eps - want| <= 2 sqrt(want) |delta| + |delta|^2 + 2^-20 want, delta_c = (D + 2) 2^-23
(|v_c| + sum |W||k|)."""
import re

import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("layers,Hkv,n_idx", [(1, 1, 1), (2, 3, 129), (1, 8, 128), (3, 2, 300), (30, 8, 700), (75, 3, 257), (151, 1, 100),
                                              (74, 1, 1), (37, 5, 300), (2, 8, 256), (20, 8, 769)])      # around where pairs of blocks begin
def test_residual_layer(oracle, layers, Hkv, n_idx):
    N, d = 800, 128
    D = Hkv * d
    gen = torch.Generator(device=DEV).manual_seed(layers * 10 + Hkv)
    K = (torch.randn(layers * Hkv, N, d, generator=gen, device=DEV) * 2).to(torch.bfloat16)
    W = (torch.randn(layers, D, D, generator=gen, device=DEV) / np.sqrt(D)).to(torch.bfloat16)
    V = torch.randn(layers * Hkv, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    idx = torch.stack([torch.randperm(N, generator=gen, device=DEV)[:n_idx].sort().values for _ in range(layers)]).to(torch.int32)
    sh = vec.Shape(1, layers, 2 * Hkv, Hkv, d, vec.VECTOR_BF16, 16)
    eps = [torch.full((layers, n_idx), float("nan"), device=DEV) for _ in range(2)]
    for e in eps:
        vec.vector_residual_layer(sh, K, V, W, N, idx, n_idx, e)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    assert torch.equal(eps[0], eps[1])
    for l in range(0, layers, max(1, layers // 5)):
        rows = idx[l].long()
        k = torch.cat([K[l * Hkv + h][rows] for h in range(Hkv)], 1).double().cpu().numpy()
        v = torch.cat([V[l * Hkv + h][rows] for h in range(Hkv)], 1).double().cpu().numpy()
        w = W[l].double().cpu().numpy()
        want = oracle.residual_layer(K[l * Hkv:(l + 1) * Hkv].cpu(), V[l * Hkv:(l + 1) * Hkv].cpu(), W[l].cpu(), idx[l].cpu().numpy())
        dn = np.sqrt((((D + 2) * 2.0 ** -23 * (np.abs(v) + np.abs(k) @ np.abs(w).T)) ** 2).sum(1))
        err = np.abs(eps[0][l].double().cpu().numpy() - want)
        assert np.all(err <= 2 * np.sqrt(want) * dn + dn ** 2 + 2.0 ** -20 * want), (l, float(err.max()))


@pytest.mark.parametrize("layers,Hkv,n_idx", [(2, 3, 129), (30, 8, 300), (37, 5, 300), (16, 8, 260)])      # two by blocks, two by pairs of blocks
def test_residual_layer_values_at_16_bytes(layers, Hkv, n_idx):
    """Values that begin at an odd multiple of 16 bytes, which is all that the interface asks for: the same residuals to the bit."""
    N, d = 400, 128
    gen = torch.Generator(device=DEV).manual_seed(7)
    K = torch.randn(layers * Hkv, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    V = torch.randn(layers * Hkv, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(layers, Hkv * d, Hkv * d, generator=gen, device=DEV) / np.sqrt(Hkv * d)).to(torch.bfloat16)
    shifted = torch.empty(V.numel() + 8, dtype=torch.bfloat16, device=DEV)[8:].view(V.shape)
    shifted.copy_(V)
    assert V.data_ptr() % 32 == 0 and shifted.data_ptr() % 32 == 16
    idx = torch.stack([torch.randperm(N, generator=gen, device=DEV)[:n_idx].sort().values for _ in range(layers)]).to(torch.int32)
    sh = vec.Shape(1, layers, 2 * Hkv, Hkv, d, vec.VECTOR_BF16, 16)
    eps = [torch.full((layers, n_idx), float("nan"), device=DEV) for _ in range(2)]
    for e, v in zip(eps, (V, shifted)):
        vec.vector_residual_layer(sh, K, v, W, N, idx, n_idx, e)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    assert torch.equal(eps[0], eps[1])


def _blocks_a_tile(layers, Hkv, n_idx):
    """Blocks that share a tile in the kernel that this call launches, by its name in a profile."""
    N, d = 2 * n_idx, 128
    K = torch.zeros(layers * Hkv, N, d, dtype=torch.bfloat16, device=DEV)
    W = torch.zeros(layers, Hkv * d, Hkv * d, dtype=torch.bfloat16, device=DEV)
    idx = torch.arange(n_idx, dtype=torch.int32, device=DEV).repeat(layers, 1).contiguous()
    eps = torch.empty(layers, n_idx, device=DEV)
    sh = vec.Shape(1, layers, Hkv, Hkv, d, vec.VECTOR_BF16, 16)
    vec.vector_residual_layer(sh, K, K, W, N, idx, n_idx, eps)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        vec.vector_residual_layer(sh, K, K, W, N, idx, n_idx, eps)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "residual_layer_tc" in e.name]
    if not names:
        pytest.skip("no kernel names from the profiler")
    return int(re.search(r"residual_layer_tc<.*?(\d)\)?>", names[0]).group(1))


def test_few_heads_and_short_lists_take_single_blocks():
    """Pairs of blocks cost 2 us before their first item: one head of 300 tokens takes 10.5 us so and 8.5 by blocks by themselves."""
    for shape in ((1, 1, 300), (16, 1, 5000), (16, 2, 5000), (1, 3, 300), (1, 4, 300)):
        assert _blocks_a_tile(*shape) == 1, shape
    for shape in ((16, 8, 5000), (1, 8, 1500), (37, 5, 1500)):
        assert _blocks_a_tile(*shape) == 2, shape
