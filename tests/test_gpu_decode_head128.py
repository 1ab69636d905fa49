"""Decode of 128-channel bf16 heads with an fp32 output: weights and key sums keep sixteen bits, without a bias.

A weight or key sum in two rounded bf16 parts is off by 2^-18.5 (2.7e-6) in the mean square and nearly unbiased; what the
heads' outputs are off by is that, once or twice over where a few keys carry the sum: at most 5e-6 in the mean square.
Where all values are one the output is the sum of the parts over the sum of the weights, in which such errors average out over
the rows to well below 1e-6; parts cut off instead of rounded would leave 2^-17.5 (5.4e-6)."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

from helpers import decode_call, decode_errors, decode_problem

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _decode(rk, rv, ak, W, q):
    U, n_ret, n_apx = q.shape[0], rk.shape[1], ak.shape[1]
    pos = [torch.zeros(U, n, dtype=torch.int32, device=DEV) for n in (n_ret, n_apx)]
    return decode_call(q, vec.Cache(rk, rv, ak, *pos, n_ret, n_apx), W, False)


@pytest.mark.parametrize("g,units,n_ret,n_apx,sharp", [(4, 4, 300, 500, 1.0), (4, 150, 300, 500, 1.0), (8, 100, 64, 700, 2.0), (1, 8, 5000, 9000, 0.2)])
def test_decode_head128_precision(oracle, g, units, n_ret, n_apx, sharp):
    q, cache, W = decode_problem(units, g, 128, torch.bfloat16, n_ret, n_apx, 31, sharp)
    errs = decode_errors(oracle, q, cache, W, decode_call(q, cache, W, False), False, range(0, units, max(1, units // 16)))
    rms = float(np.sqrt(np.mean(errs ** 2)))
    assert rms <= 5e-6, rms


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("units,n_ret", [(8, 2457), (600, 512)])
def test_decode_of_equal_values(d, units, n_ret):
    gen = torch.Generator(device=DEV).manual_seed(37)
    rk = torch.randn(units, n_ret, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = torch.eye(d, device=DEV).repeat(units, 1, 1).to(torch.bfloat16)
    q = (torch.randn(units, 4, d, generator=gen, device=DEV) * 0.3).to(torch.bfloat16)
    out = _decode(rk, torch.ones_like(rk), torch.zeros(units, 0, d, dtype=torch.bfloat16, device=DEV), W, q)
    assert (out.double() - 1).pow(2).mean().sqrt().item() <= 1e-6


def _rising(U, n, rises, gen, q):
    """Keys of which one in each of len(rises) equal spans has the logit rises[i] (in powers of two) against q, the rest -60 or less."""
    d, span = q.shape[-1], n // len(rises)
    level = torch.full((U, n), -60.0, device=DEV)
    for i, r in enumerate(rises):
        at = torch.randint(0, span, (U,), generator=gen, device=DEV) + i * span
        level.scatter_(1, at[:, None], r + torch.rand(U, 1, generator=gen, device=DEV) * 0.3)
    return (level[..., None] * np.log(2.0) * q.float()[:, None, :] / np.sqrt(d)).to(torch.bfloat16)


def _unit_queries(U, d, gen):
    q = torch.randn(U, d, generator=gen, device=DEV)
    return (q / q.norm(dim=1, keepdim=True) * np.sqrt(d)).to(torch.bfloat16)


def _largest_weight_exact(q, rk, rv, out):
    """The weight that carries the sum must not be rounded: were it, it would leave 2^-18.5 of the output (2.7e-6) in the mean square."""
    p = torch.softmax(torch.einsum("ud,und->un", q.double(), rk.double()) / np.sqrt(q.shape[-1]), 1)
    o = torch.einsum("un,und->ud", p, rv.double())
    err = ((out.double() - o).norm(dim=1) / o.norm(dim=1)).pow(2).mean().sqrt().item()
    assert err <= 1e-6, err


@pytest.mark.parametrize("units", [2000])
def test_decode_head128_largest_weight(units):
    """Six tiles of 64 rows a unit, whose maxima rise by 2.5 powers of two: a warp has two of them, three apart."""
    d, gen = 128, torch.Generator(device=DEV).manual_seed(41)
    q = _unit_queries(units, d, gen)
    rk, rv = _rising(units, 384, [2.5 * i for i in range(6)], gen, q), torch.randn(units, 384, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = torch.zeros(units, d, d, dtype=torch.bfloat16, device=DEV)
    out = _decode(rk, rv, torch.zeros(units, 0, d, dtype=torch.bfloat16, device=DEV), W, q[:, None, :].contiguous())
    _largest_weight_exact(q, rk, rv, out[:, 0])


def test_decode_layer_largest_weight():
    """Three tiles of 16 tokens a (sequence, layer), whose maxima rise by 3.9 powers of two."""
    d, Hkv, layers, gen = 128, 8, 148, torch.Generator(device=DEV).manual_seed(43)
    U = Hkv * layers
    q = _unit_queries(U, d, gen)
    rk, rv = _rising(U, 48, [0.0, 3.7, 7.4], gen, q), torch.randn(U, 48, d, generator=gen, device=DEV).to(torch.bfloat16)
    W = torch.zeros(layers, Hkv * d, Hkv * d, dtype=torch.bfloat16, device=DEV)
    sh = vec.Shape(1, layers, Hkv, Hkv, d, vec.VECTOR_BF16, 16)
    pos = [torch.zeros(U, n, dtype=torch.int32, device=DEV) for n in (48, 0)]
    cache = vec.Cache(rk, rv, torch.zeros(U, 0, d, dtype=torch.bfloat16, device=DEV), *pos, 48, 0)
    ws = torch.empty(vec.vector_layer_workspace_bytes(sh, vec.vector_plan_budget(8192, 4096, -1, 16)), dtype=torch.uint8, device=DEV)
    out = torch.full((U, 1, d), float("nan"), device=DEV)
    vec.vector_decode_attn_layer(sh, q[:, None, :].contiguous(), cache, W, out, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    _largest_weight_exact(q, rk, rv, out[:, 0])
