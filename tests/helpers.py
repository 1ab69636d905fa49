"""Shared helpers of the parity tests: run the oracle unit by unit on the exact stored bits."""
import numpy as np
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200 import synth


def shape_of(wl, batch=None, n_layers=None):
    return vec.Shape(wl.batch if batch is None else batch, wl.n_layers if n_layers is None else n_layers,
                     wl.n_q_heads, wl.n_kv_heads, wl.head_dim,
                     vec.VECTOR_BF16 if wl.dtype == "bf16" else vec.VECTOR_F32, wl.window, wl.pool_kernel)


def budget_of(wl, percent, n_a=-1):
    return vec.vector_plan_budget(wl.N, (wl.N * percent) // 100, n_a, wl.window)


def calibrated_maps(wl, device="cuda"):
    """W [LH][d][d] in the workload dtype (the bits both sides use), via the library's host solver.
    `device` is where the calibration draw is generated: it must be the device the context tensors are
    generated on, because the per-head parameters (channel scales, true map) come from that device's
    random stream."""
    from paper_2605_23258_b200.pipeline import calibrate_maps
    pairs = []
    for l in range(wl.n_layers):
        for h in range(wl.n_kv_heads):
            k, v = synth.calib_kv(wl, l, h, device)
            pairs.append((k.cpu(), v.cpu()))
    return calibrate_maps(pairs, wl.lam).to(wl.torch_dtype)


def oracle_scores(oracle, wl, Q, K):
    """Q [U][g][w][d], K [U][N][d] (cpu) -> raw, score float64 [U][N]."""
    scale = 1.0 / np.sqrt(wl.head_dim)
    raws, scs = [], []
    for u in range(K.shape[0]):
        r, s = oracle.score(Q[u], K[u], scale, wl.pool_kernel)
        raws.append(r), scs.append(s)
    return np.stack(raws), np.stack(scs)


def score_close(got, want, mass, rtol=1e-3):
    """|g - o| <= rtol * max(|o|, 1e-6 * mass) elementwise on the finite entries; infinities must match."""
    got, want = np.asarray(got, np.float64), np.asarray(want, np.float64)
    inf_ok = np.array_equal(np.isinf(got), np.isinf(want)) and np.all(got[np.isinf(got)] > 0)
    fin = np.isfinite(want)
    err = np.abs(got[fin] - want[fin])
    tol = rtol * np.maximum(np.abs(want[fin]), 1e-6 * mass)
    return inf_ok and bool(np.all(err <= tol)), float(np.max(err / tol)) if err.size else 0.0


def eps_close(got, want, K_rows, V_rows, W):
    """Residual eps = sum_c r_c^2, r = v - W k, computed on the device with fp32 accumulation of exact
    bf16/fp32 products against the oracle's fp64.  Each r_c carries an absolute error of at most
    delta_c = 130 * 2^-23 * (|v_c| + sum_j |W_cj| |k_j|)   (d + 2 roundings of relative size 2^-23, a
    bound that also covers an accumulator that truncates instead of rounding), so
    |eps_gpu - eps| <= 2 sqrt(eps) ||delta|| + ||delta||^2, plus 2^-21 eps for the fp32 sum of squares."""
    K_rows, V_rows, W = (np.asarray(t.double().numpy() if hasattr(t, "double") else t, np.float64) for t in (K_rows, V_rows, W))
    delta = 130 * 2.0 ** -23 * (np.abs(V_rows) + np.abs(K_rows) @ np.abs(W).T)
    dn = np.sqrt((delta ** 2).sum(1))
    want = np.asarray(want, np.float64)
    tol = 2 * np.sqrt(want) * dn + dn ** 2 + 2.0 ** -21 * want
    err = np.abs(np.asarray(got, np.float64) - want)
    return bool(np.all(err <= tol)), float(np.max(err / tol))


def decode_problem(U, g, d, dtype, n_ret, n_apx, seed, sharp=1.0, device="cuda"):
    """Random pools with two rows to spare, a map per unit and queries.  In both pools the first and last row and the rows on
    either side of every 64th get a key towards the unit's first query, so that each of them carries a visible share of the output:
    losing one shows as a thousandth of it or more."""
    gen = torch.Generator(device=device).manual_seed(seed)
    q = (torch.randn(U, g, d, generator=gen, device=device) * sharp).to(dtype)
    unit = q[:, :1].float() / q[:, :1].float().norm(dim=-1, keepdim=True)

    def keys(n):
        k = torch.randn(U, n + 2, d, generator=gen, device=device)
        rows = sorted({r for r in (0, n - 1, *range(63, n, 64), *range(64, n, 64)) if 0 <= r < n})
        if rows:
            k[:, rows] += 4.0 / sharp * unit
        return k.to(dtype)
    rk, ak = keys(n_ret), keys(n_apx)
    rv = torch.randn(U, n_ret + 2, d, generator=gen, device=device).to(dtype)
    W = (torch.randn(U, d, d, generator=gen, device=device) / np.sqrt(d)).to(dtype)
    pos = torch.randint(0, 131072, (U, n_apx + 2), generator=gen, device=device, dtype=torch.int32)
    ret_pos = torch.zeros(U, n_ret + 2, dtype=torch.int32, device=device)
    return q, vec.Cache(rk, rv, ak, ret_pos, pos, n_ret, n_apx), W


def decode_shape(q, rope):
    U, g, d = q.shape
    return vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16 if q.dtype == torch.bfloat16 else vec.VECTOR_F32, 16, 7, 0.0, int(rope), 10000.0)


def decode_call(q, cache, W, rope, out_dtype=torch.float32, mode=0, times=1):
    sh = decode_shape(q, rope)
    out = torch.full(q.shape, float("nan"), dtype=out_dtype, device=q.device)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(16384, 8192, -1, 16))
    for _ in range(times):
        vec.vector_decode_attn(sh, q, cache, W, out, mode, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    return out


def decode_errors(oracle, q, cache, W, out, rope, units):
    """Per head of the listed units: the 2-norm of what the output is off by, over the output's."""
    errs = []
    for u in units:
        _, o = oracle.attend(q[u].cpu(), cache.ret_k[u, :cache.n_ret].cpu(), cache.ret_v[u, :cache.n_ret].cpu(), cache.apx_k[u, :cache.n_apx].cpu(),
                             W[u].cpu(), 1.0 / np.sqrt(q.shape[-1]), apx_pos=cache.apx_pos[u, :cache.n_apx].cpu().numpy(), rope=rope, theta=10000.0)
        errs.append(np.linalg.norm(out[u].cpu().double().numpy() - o, axis=1) / np.linalg.norm(o, axis=1))
    return np.concatenate(errs)


def decode_bound(dtype, d, rope):
    """What an fp32 output may be off by, per head.  fp32 keys, and 64-channel bf16 heads: a few roundings of exponentials (2^-22) and
    logits (|s| 2^-24, |s| up to 20), 3e-6.  128-channel bf16 heads: weights and key sums in two bf16 parts, 2^-17 each of a head that
    one row may carry, 1.5e-5; keys turned back as fp16, 2^-12 each, whose sum may cancel to a third, 8e-4."""
    if dtype == torch.float32 or d == 64:
        return 3e-6
    return 8e-4 if rope else 1.5e-5
