"""The fp32 kernels at the sizes where their launches change: normalisers formed inline or by a kernel of their own, ragged
tiles, clusters of one to sixteen blocks, two or four residual rows a warp.  Scores 1e-3 relative (score_close), residuals within
the rounding bound (eps_close), attention to helpers.decode_bound, 2^-8 more for a bf16 output."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import synth

from helpers import decode_bound, decode_call, decode_errors, decode_problem, eps_close, oracle_scores, score_close, shape_of

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("N,d,heads,g,window", [(64, 64, 1, 1, 64), (65, 128, 2, 3, 50), (2048, 64, 1, 2, 33), (2049, 128, 1, 8, 25), (5000, 64, 3, 1, 16)])
def test_score_fp32(oracle, N, d, heads, g, window):
    wl = synth.shrink(synth.WORKLOADS[0], N=N, head_dim=d, n_kv_heads=heads, n_q_heads=heads * g, window=window)
    K, _, Q = synth.context(wl, DEV)
    scores = torch.empty(wl.units, N, device=DEV)
    vec.vector_score(shape_of(wl), Q, K, N, scores, None, vec.alloc_workspace(shape_of(wl), vec.vector_plan_budget(N, N, 0, window)))
    torch.cuda.synchronize()
    _, want = oracle_scores(oracle, wl, Q.cpu(), K.cpu())
    ok, worst = score_close(scores.cpu().numpy(), want, g * window)
    assert ok, f"score off by {worst:.3g} x tolerance"


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("U,n_idx", [(1, 1), (3, 17), (40, 129)])
def test_residual_fp32(oracle, rope, d, U, n_idx):
    gen = torch.Generator(device=DEV).manual_seed(U)
    K, V = (torch.randn(U, 300, d, generator=gen, device=DEV) for _ in range(2))
    W = torch.randn(U, d, d, generator=gen, device=DEV) / np.sqrt(d)
    idx = torch.stack([torch.randperm(300, generator=gen, device=DEV)[:n_idx].sort().values for _ in range(U)]).to(torch.int32)
    sh = vec.Shape(1, 1, U, U, d, vec.VECTOR_F32, 16, 7, 0.0, int(rope), 10000.0)
    eps = torch.full((U, n_idx), float("nan"), device=DEV)
    vec.vector_residual(sh, K, V, W, 300, idx, n_idx, eps)
    torch.cuda.synchronize()
    for u in range(0, U, max(1, U // 4)):
        rows = idx[u].long().cpu()
        want = oracle.residual(K[u].cpu(), V[u].cpu(), W[u].cpu(), idx[u].cpu().numpy(), rope=rope, theta=10000.0)
        ok, worst = eps_close(eps[u].cpu().numpy(), want, K[u].cpu()[rows], V[u].cpu()[rows], W[u].cpu())
        assert ok, f"unit {u}: eps off by {worst:.3g} x bound"


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("d,U,g,n_ret,n_apx", [(64, 1, 1, 1, 0), (64, 2, 8, 0, 31), (128, 3, 2, 33, 32), (128, 1, 5, 700, 900), (64, 300, 4, 40, 70)])
def test_decode_fp32(oracle, rope, d, U, g, n_ret, n_apx):
    q, cache, W = decode_problem(U, g, d, torch.float32, n_ret, n_apx, U + g, sharp=2.0)
    units = range(0, U, max(1, U // 4))
    bound = decode_bound(torch.float32, d, rope)
    for out_dtype, more in ((torch.float32, 0.0), (torch.bfloat16, 2.0 ** -8)):
        errs = decode_errors(oracle, q, cache, W, decode_call(q, cache, W, rope, out_dtype), rope, units)
        assert errs.max() <= bound + more, errs.max()
