"""The allocation-free decode entry point against the workspace-taking one.

vector_decode_attn_static serves callers that cannot allocate device memory at
call time (a server whose own pool holds the whole device, or a decode loop that
cannot afford a cudaMalloc stall): its split-KV scratch is a fixed array inside
the library.  It must give what vector_decode_attn gives, call after call, since
every call reuses the same array with the previous call's contents still in it.
This file sorts last so that a run that stops at the first failure has already
run every other test.
"""
import gc

import pytest
import torch

import paper_2605_23258_b200 as vec

pytestmark = pytest.mark.gpu
DEV = "cuda"
# More units than the one-launch form takes, so that records go through the array; the one-launch form and fp32 write none.
STREAM_UNITS = 80


def _problem(U, g, d, dtype, rope, n_ret, n_apx, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rk, rv = (torch.randn(U, n_ret, d, generator=gen, device=DEV).to(dtype) for _ in range(2))
    ak = torch.randn(U, n_apx, d, generator=gen, device=DEV).to(dtype)
    W = (torch.randn(U, d, d, generator=gen, device=DEV) / d ** 0.5).to(dtype)
    q = torch.randn(U, g, d, generator=gen, device=DEV).to(dtype)
    pos = [torch.randint(0, 4096, (U, n), generator=gen, device=DEV, dtype=torch.int32) for n in (n_ret, n_apx)]
    sh = vec.Shape(1, 1, U * g, U, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, 16, 7, 0.0, int(rope), 10000.0)
    assert 0 < vec.vector_decode_scratch_bytes(sh) <= vec.VECTOR_STATIC_SCRATCH_BYTES
    return sh, q, vec.Cache(rk, rv, ak, *pos, n_ret, n_apx), W


def _launches(call):
    before = vec.vector_kernel_launches()
    call()
    return vec.vector_kernel_launches() - before


@pytest.mark.parametrize("d,g,rope,mode", [(128, 4, False, 0), (128, 8, False, 1), (64, 3, False, 0), (128, 2, True, 0), (64, 8, True, 0)])
def test_static_scratch_decode_matches_workspace_decode_twice(d, g, rope, mode):
    # two calls in a row on different problems: the second finds the first one's records in the array
    for step, (n_ret, n_apx) in enumerate([(300, 521), (700, 129)]):
        sh, q, cache, W = _problem(STREAM_UNITS, g, d, torch.bfloat16, rope, n_ret, n_apx, step)
        ws = vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16))
        for dt in (torch.float32, torch.bfloat16):
            want = torch.empty(STREAM_UNITS, g, d, dtype=dt, device=DEV)
            got = torch.full_like(want, float("nan"))
            vec.vector_decode_attn(sh, q, cache, W, want, mode, ws)
            # a streaming kernel, whose records the merge kernel reads: without records this test would check nothing
            assert _launches(lambda: vec.vector_decode_attn_static(sh, q, cache, W, got, mode)) == 2
            torch.cuda.synchronize()
            assert torch.isfinite(got).all()
            assert torch.equal(got, want)          # same kernels, same launch shape, same inputs


def test_static_scratch_all_record_layouts_back_to_back_and_no_allocation():
    """Records differ with the head size, the heads a unit has, the warps that write them (four, three, or two with values
    rebuilt tile by tile) and RoPE: the calls run in turn, so that each finds the others' leftovers, with a one-launch and an fp32 call,
    which leave none, among them; and no call takes device memory (free bytes of the device and the bytes torch holds unchanged)."""
    bf16 = torch.bfloat16
    forms = [(STREAM_UNITS, 4, 128, bf16, False, 0, 2), (STREAM_UNITS, 8, 64, bf16, False, 0, 2), (STREAM_UNITS, 4, 128, bf16, False, 1, 2),
             (STREAM_UNITS, 2, 128, bf16, True, 0, 2), (4, 4, 128, bf16, False, 0, 1), (STREAM_UNITS, 5, 64, bf16, True, 0, 2),
             (2, 2, 64, torch.float32, False, 0, 1)]
    cases = []
    for i, (U, g, d, dtype, rope, mode, kernels) in enumerate(forms):
        sh, q, cache, W = _problem(U, g, d, dtype, rope, 200 + 64 * i, 400 - 50 * i, i)
        want = torch.empty(U, g, d, dtype=torch.float32, device=DEV)
        vec.vector_decode_attn(sh, q, cache, W, want, mode, vec.alloc_workspace(sh, vec.vector_plan_budget(4096, 2048, -1, 16)))
        cases.append((sh, q, cache, W, want, mode, kernels))
    for sh, q, cache, W, want, mode, kernels in cases:         # the first call per device looks the array up
        out = torch.empty_like(want)
        assert _launches(lambda: vec.vector_decode_attn_static(sh, q, cache, W, out, mode)) == kernels
    rounds = [[torch.full_like(c[4], float("nan")) for c in cases] for _ in range(3)]
    gc.collect()                                               # tensors of earlier tests must not be released in between
    torch.cuda.synchronize()
    free0, held0 = torch.cuda.mem_get_info()[0], torch.cuda.memory_allocated()
    for outs in rounds:                                        # nothing but the library's calls in between
        for case, o in zip(cases, outs):
            vec.vector_decode_attn_static(case[0], case[1], case[2], case[3], o, case[5])
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free0 and torch.cuda.memory_allocated() == held0
    for outs in rounds:
        for case, o in zip(cases, outs):
            assert torch.equal(o, case[4])


def test_static_scratch_rejects_shapes_beyond_its_limit():
    # 65535 units of 8 query heads need far more partial records than the fixed array holds
    big = vec.Shape(1, 1, 8 * 65535, 65535, 128, vec.VECTOR_BF16, 64)
    assert vec.vector_decode_scratch_bytes(big) > vec.VECTOR_STATIC_SCRATCH_BYTES
    t = torch.zeros(16, dtype=torch.bfloat16, device=DEV)
    i = torch.zeros(16, dtype=torch.int32, device=DEV)
    cache = vec.Cache(t.view(1, 1, 16), t.view(1, 1, 16), t.view(1, 1, 16), i.view(1, 16), i.view(1, 16), 1, 0)
    with pytest.raises(vec.VectorError) as e:
        vec.vector_decode_attn_static(big, t, cache, t, torch.zeros(16, device=DEV))
    assert e.value.status == -5
