"""Scores of units with few rows (up to 128 have kernels of their own) and of few units (pooled by the second pass), around the sizes
where a tile, a chunk or a group of rows ends, windows narrower than the pooling radius among them; many units with the same
shapes take the other route and give the same scores.  Bound, as for every score test: 1e-3 of the value or of 1e-6 of the mass."""
import pytest
import torch

import paper_2605_23258_b200 as vec
from helpers import score_close

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("units", [1, 3, 150])
@pytest.mark.parametrize("d,g,w,N,pool", [
    (128, 1, 16, 2049, 7), (128, 3, 32, 5000, 7), (64, 1, 100, 1401, 7), (64, 8, 16, 3071, 15), (128, 2, 64, 640, 1), (128, 1, 1, 130, 15),
    (64, 1, 2, 257, 15), (128, 1, 129, 1000, 7), (64, 4, 64, 4097, 7), (128, 4, 48, 1281, 5), (128, 3, 100, 1500, 7), (128, 2, 3, 128, 7)])
def test_score(oracle, units, d, g, w, N, pool):
    gen = torch.Generator(device=DEV).manual_seed(d + g + w + N)
    K = torch.randn(units, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    Q = (torch.randn(units, g, w, d, generator=gen, device=DEV) * 2).to(torch.bfloat16)
    sh = vec.Shape(1, units, g, 1, d, vec.VECTOR_BF16, w, pool)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(N, N, 0, w))
    scores, raw, again = (torch.full((units, N), float("nan"), device=DEV) for _ in range(3))
    vec.vector_score(sh, Q, K, N, scores, raw, ws)
    vec.vector_score(sh, Q, K, N, again, None, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    assert torch.equal(scores, again)
    for u in sorted({0, units // 2, units - 1}):
        raw_o, sc_o = oracle.score(Q[u].cpu(), K[u].cpu(), d ** -0.5, pool)
        for got, want in ((raw[u], raw_o), (scores[u], sc_o)):
            ok, worst = score_close(got.cpu().numpy()[None], want[None], g * w)
            assert ok, (u, worst)


@pytest.mark.parametrize("units,d,g,w,N,pool", [
    (1, 64, 1, 16, 65, 1), (2, 64, 2, 3, 64 - 14 + 1, 15), (2, 128, 1, 2, 2 * (64 - 14) + 1, 15), (1, 128, 3, 1, 1, 15), (1, 64, 1, 5, 6, 15),
    (2, 128, 4, 32, 2 * (64 - 6) + 1, 7), (1, 128, 2, 50, 58, 7), (1, 64, 5, 20, 20, 15), (1, 64, 2, 40, 2047, 1),
    (150, 64, 1, 32, 300, 7), (130, 64, 5, 16, 300, 15), (40, 64, 1, 70, 1100, 1), (2, 64, 8, 100, 4000, 5), (150, 128, 1, 32, 290, 7)])
def test_score_fp32(oracle, units, d, g, w, N, pool):
    """fp32 on CUDA cores: lengths that end one key into a tile, windows narrower than the pooling radius, pools of one key; so few tiles
    that the second pass pools them, and more blocks than four a multiprocessor.  Raw sums asked for or not."""
    gen = torch.Generator(device=DEV).manual_seed(d + g + w + N)
    K = torch.randn(units, N, d, generator=gen, device=DEV)
    Q = torch.randn(units, g, w, d, generator=gen, device=DEV) * 2
    sh = vec.Shape(1, units, g, 1, d, vec.VECTOR_F32, w, pool)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(N, N, 0, w))
    scores, raw, again = (torch.full((units, N), float("nan"), device=DEV) for _ in range(3))
    vec.vector_score(sh, Q, K, N, scores, raw, ws)
    vec.vector_score(sh, Q, K, N, again, None, ws)
    torch.cuda.synchronize()
    assert torch.equal(scores, again)
    for u in sorted({0, units // 2, units - 1}):
        raw_o, sc_o = oracle.score(Q[u].cpu(), K[u].cpu(), d ** -0.5, pool)
        for got, want in ((raw[u], raw_o), (scores[u], sc_o)):
            ok, worst = score_close(got.cpu().numpy()[None], want[None], g * w)
            assert ok, (u, worst)


@pytest.mark.parametrize("d,rows", [(128, 96), (128, 300), (64, 96)])
def test_workspace_is_enough(d, rows):
    """With little to select, the scores' sums are what the workspace is sized by: nothing is written behind it."""
    U, N = 200, 20000
    gen = torch.Generator(device=DEV).manual_seed(rows)
    K = torch.randn(U, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    Q = torch.randn(U, 1, rows, d, generator=gen, device=DEV).to(torch.bfloat16)
    sh = vec.Shape(1, U, 1, 1, d, vec.VECTOR_BF16, rows)
    need = vec.vector_workspace_bytes(sh, vec.vector_plan_budget(N, 512, -1, rows))
    room = torch.full((need + 65536,), 7, dtype=torch.uint8, device=DEV)
    got, want = (torch.full((U, N), float("nan"), device=DEV) for _ in range(2))
    vec.vector_score(sh, Q, K, N, got, None, room[:need])
    vec.vector_score(sh, Q, K, N, want, None, torch.empty(2 * need, dtype=torch.uint8, device=DEV))
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    assert torch.equal(got, want) and bool((room[need:] == 7).all())
