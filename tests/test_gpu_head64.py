"""bf16 with 64-channel heads on the tensor-core kernels: sizes at the edges of their tiles against the oracle.

Scores 1e-3 relative (score_close); residuals within the rounding bound of fp32 accumulation (eps_close);
attention 2e-2 absolute in fp32 output, the tolerances of the 128-channel kernels."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import synth

from helpers import budget_of, calibrated_maps, decode_call, decode_errors, decode_problem, eps_close, oracle_scores, score_close, shape_of

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _workload(**over):
    return synth.shrink(synth.WORKLOADS[1], head_dim=64, n_calib=512, **over)


@pytest.mark.parametrize("over", [
    {"N": 128, "n_kv_heads": 1, "n_q_heads": 1, "window": 16},                    # one tile, one row block
    {"N": 2 * 1024 + 129, "n_kv_heads": 2, "n_q_heads": 16, "window": 128},       # 1024 rows: four row groups; the key ring wraps
    {"N": 1300, "n_layers": 20, "n_kv_heads": 8, "n_q_heads": 24, "window": 50},  # several items per block, 150 rows, ragged end
])
def test_score_head64(oracle, over):
    wl = _workload(**over)
    K, _, Q = synth.context(wl, DEV)
    sh = shape_of(wl)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(wl.N, wl.N, 0, wl.window))
    scores = torch.empty(wl.units, wl.N, dtype=torch.float32, device=DEV)
    raw = torch.empty_like(scores)
    vec.vector_score(sh, Q, K, wl.N, scores, raw, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    mass = wl.group * wl.window
    assert np.allclose(raw.double().sum(1).cpu().numpy(), mass, rtol=1e-4)
    units = list(range(wl.units))[:: max(1, wl.units // 6)]
    raw_o, sc_o = oracle_scores(oracle, wl, Q[units].cpu(), K[units].cpu())
    for got, want in ((scores, sc_o), (raw, raw_o)):
        ok, worst = score_close(got[units].cpu().numpy(), want, mass)
        assert ok, f"off by {worst:.3g} x tolerance"


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("n_idx,layers", [(1, 1), (129, 1), (700, 40)])           # a row, a tile and a row, rings that wrap over units
def test_residual_head64(oracle, rope, n_idx, layers):
    wl = _workload(N=900, n_kv_heads=2, n_q_heads=4, n_layers=layers)
    K, V, _ = synth.context(wl, DEV)
    if rope:
        K = synth.rope_keys(K)
    W = calibrated_maps(wl).to(DEV)
    sh = shape_of(wl)
    sh.rope_enabled = int(rope)
    g = torch.Generator().manual_seed(5)
    idx = torch.stack([torch.randperm(wl.N, generator=g)[:n_idx].sort().values for _ in range(wl.units)]).to(torch.int32).to(DEV)
    eps = torch.full((wl.units, n_idx), float("nan"), device=DEV)
    vec.vector_residual(sh, K, V, W, wl.N, idx, n_idx, eps)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    for u in range(0, wl.units, max(1, wl.units // 8)):
        Kc, Vc, Wc, rows = K[u].cpu(), V[u].cpu(), W[u % W.shape[0]].cpu(), idx[u].long().cpu()
        want = oracle.residual(Kc, Vc, Wc, idx[u].cpu().numpy(), rope=rope, theta=sh.rope_theta)
        ok, worst = eps_close(eps[u].cpu().numpy(), want, Kc[rows], Vc[rows], Wc)
        assert ok, f"unit {u}: eps off by {worst:.3g} x bound"


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("g,layers,n_ret,n_apx", [
    (1, 1, 1, 0), (2, 1, 0, 65), (4, 1, 64, 128), (8, 1, 1000, 3000 + 7),         # a key, half a tile, whole tiles, long ranges
    (3, 40, 130, 257),                                                            # many units: ranges cross unit ends
])
def test_decode_head64(oracle, rope, g, layers, n_ret, n_apx):
    wl = _workload(N=4096, n_kv_heads=2, n_q_heads=2 * g, n_layers=layers)
    U, d = wl.units, wl.head_dim
    gen = torch.Generator(device=DEV).manual_seed(9)
    rk, rv = (torch.randn(U, n_ret + 1, d, generator=gen, device=DEV).to(torch.bfloat16) for _ in range(2))
    ak = torch.randn(U, n_apx + 3, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(2 * layers, d, d, generator=gen, device=DEV) / 8).to(torch.bfloat16)
    q = (torch.randn(U, g, d, generator=gen, device=DEV) * 2).to(torch.bfloat16)
    pos = torch.randint(0, 131072, (U, n_apx + 3), generator=gen, device=DEV, dtype=torch.int32)
    cache = vec.Cache(rk, rv, ak, torch.zeros(U, n_ret + 1, dtype=torch.int32, device=DEV), pos, n_ret, n_apx)
    sh = shape_of(wl)
    sh.rope_enabled = int(rope)
    out = torch.full((U, g, d), float("nan"), device=DEV)
    vec.vector_decode_attn(sh, q, cache, W, out, 0, vec.alloc_workspace(sh, budget_of(wl, 50)))
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    for u in range(0, U, max(1, U // 8)):
        _, o = oracle.attend(q[u].cpu(), rk[u, :n_ret].cpu(), rv[u, :n_ret].cpu(), ak[u, :n_apx].cpu(), W[u % W.shape[0]].cpu(),
                             1.0 / np.sqrt(d), apx_pos=pos[u, :n_apx].cpu().numpy(), rope=rope, theta=sh.rope_theta)
        assert np.max(np.abs(out[u].cpu().double().numpy() - o)) <= 2e-2, u


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("g,units,n_ret,n_apx,sharp", [
    (4, 4, 70, 140, 2.0), (8, 4, 70, 140, 2.0),               # the one-launch form: third parts in spare rows, or in a fragment of their own
    (4, 80, 70, 140, 2.0), (5, 80, 70, 140, 2.0),             # records and merge
    (3, 80, 0, 300, 2.0), (1, 2, 3000, 6000, 0.3),            # key-only tiles alone; long sums of nearly equal weights
])
def test_decode_head64_keeps_fp32_precision(oracle, rope, g, units, n_ret, n_apx, sharp):
    """fp32 output to fp32's own precision, as CUDA cores give it: weights and sums that keep only sixteen bits are off by
    1e-6 and more.  What remains is the exponentials' 2^-22 and the logits' rounding, |s| 2^-24 a few times over with |s| up to
    20: at most about 1e-6 in a head, and less than half of that in the mean square over the heads."""
    q, cache, W = decode_problem(units, g, 64, torch.bfloat16, n_ret, n_apx, 17, sharp)
    errs = decode_errors(oracle, q, cache, W, decode_call(q, cache, W, rope), rope, range(0, units, max(1, units // 16)))
    assert errs.max() <= 1.5e-6 and np.sqrt(np.mean(errs ** 2)) <= 5e-7, (errs.max(), np.sqrt(np.mean(errs ** 2)))


def test_decode_head64_rope_keeps_large_keys(oracle):
    """Keys beyond the fp16 range, and positions of either sign: a turned key keeps bf16's range."""
    U, g, d, n = 3, 4, 64, 100
    gen = torch.Generator(device=DEV).manual_seed(3)
    ak = (torch.randn(U, n, d, generator=gen, device=DEV) * 3e5).to(torch.bfloat16)
    rk, rv = (torch.zeros(U, 1, d, dtype=torch.bfloat16, device=DEV) for _ in range(2))
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / 8).to(torch.bfloat16)
    q = (torch.randn(U, g, d, generator=gen, device=DEV) * 1e-6).to(torch.bfloat16)
    pos = torch.randint(-131072, 131072, (U, n), generator=gen, device=DEV, dtype=torch.int32)
    cache = vec.Cache(rk, rv, ak, torch.zeros(U, 1, dtype=torch.int32, device=DEV), pos, 0, n)
    sh = vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16, 16, 7, 0.0, 1, 10000.0)
    out = torch.full((U, g, d), float("nan"), device=DEV)
    vec.vector_decode_attn(sh, q, cache, W, out, 0, vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16)))
    torch.cuda.synchronize()
    for u in range(U):
        _, o = oracle.attend(q[u].cpu(), rk[u, :0].cpu(), rv[u, :0].cpu(), ak[u].cpu(), W[u].cpu(), 1.0 / np.sqrt(d),
                             apx_pos=pos[u].cpu().numpy(), rope=True, theta=10000.0)
        err = np.linalg.norm(out[u].cpu().double().numpy() - o, axis=1) / np.linalg.norm(o, axis=1)
        assert err.max() <= 3e-6, err


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("units,n_idx", [(3, 129), (200, 700)])
def test_residual_head64_keeps_fp32_precision(oracle, rope, units, n_idx):
    """Residuals of values that the map nearly gives: (eps - want) / (2 sqrt(want)) is the error of W k~ along the residual.
    fp32 leaves a few 2^-24 of the prediction's size, keys kept to 2^-17 about 2^-18.5 of it: at most 2^-22 in the mean square."""
    d, N = 64, 900
    gen = torch.Generator(device=DEV).manual_seed(23)
    K = torch.randn(units, N, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = (torch.randn(units, d, d, generator=gen, device=DEV) / 8).to(torch.bfloat16)
    k = K.double()
    if rope:                                                  # turned back by the token's index
        angle = torch.arange(N, device=DEV).double()[:, None] * 10000.0 ** (-2.0 * torch.arange(d // 2, device=DEV).double() / d)
        cs, sn, x, y = torch.cos(angle), torch.sin(angle), k[..., :d // 2], k[..., d // 2:]
        k = torch.cat([x * cs + y * sn, y * cs - x * sn], dim=-1)
    pred = torch.bmm(k, W.double().transpose(1, 2))
    V = (pred + 0.05 * torch.randn(units, N, d, generator=gen, device=DEV)).to(torch.bfloat16)
    idx = torch.stack([torch.randperm(N, generator=gen, device=DEV)[:n_idx].sort().values for _ in range(units)]).to(torch.int32)
    sh = vec.Shape(1, 1, units, units, d, vec.VECTOR_BF16, 16, 7, 0.0, int(rope), 10000.0)
    eps = torch.full((units, n_idx), float("nan"), device=DEV)
    vec.vector_residual(sh, K, V, W, N, idx, n_idx, eps)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    errs = []
    for u in range(0, units, max(1, units // 8)):
        want = oracle.residual(K[u].cpu(), V[u].cpu(), W[u].cpu(), idx[u].cpu().numpy(), rope=rope, theta=10000.0)
        errs.append((eps[u].cpu().double().numpy() - want) / (2 * np.sqrt(want)))
    rms = float(np.sqrt(np.mean(np.concatenate(errs) ** 2)) / pred.pow(2).mean().sqrt())
    assert rms <= 2.0 ** -22, rms
