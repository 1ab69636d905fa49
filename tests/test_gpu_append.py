"""Appending a generated token: the rows, their neighbours and the positions, bit for bit, for every row width; and inputs
that are assigned rather than copied (another type, broadcast, strided, off a 16-byte boundary)."""
import pytest
import torch

import paper_2605_23258_b200 as vec
from paper_2605_23258_b200.pipeline import Compressor

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.float32, 128), (torch.bfloat16, 64), (torch.bfloat16, 128)])
@pytest.mark.parametrize("U", [1, 3, 130])
def test_append_rows(dtype, d, U):
    sh = vec.Shape(1, 1, U, U, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, 16)
    comp = Compressor(sh, vec.vector_plan_budget(200, 60, 10, 16), extra_rows=3)
    c, n = comp.cache, comp.cache.n_ret
    gen = torch.Generator(device=DEV).manual_seed(U)
    for t in (c.ret_k, c.ret_v):
        t.copy_(torch.randn(t.shape, generator=gen, device=DEV))
    c.ret_pos.fill_(-7)
    want = [t.clone() for t in (c.ret_k, c.ret_v, c.ret_pos)]
    steps = [(torch.randn(U, d, generator=gen, device=DEV).to(dtype), torch.randn(U, d, generator=gen, device=DEV).to(dtype), 2**31 - 1),
             (torch.randn(U, d, generator=gen, device=DEV, dtype=torch.float64), torch.randn(1, d, generator=gen, device=DEV), 11),
             (torch.randn(d, U, generator=gen, device=DEV).to(dtype).T, torch.randn(U, d, generator=gen, device=DEV).to(dtype), 12)]
    for i, (k, v, pos) in enumerate(steps):
        comp.append(k, v, pos)
        want[0][:, n + i], want[1][:, n + i], want[2][:, n + i] = k, v, pos
    torch.cuda.synchronize()
    assert c.n_ret == n + 3
    for got, w in zip((c.ret_k, c.ret_v, c.ret_pos), want):
        assert torch.equal(got, w)
    with pytest.raises(ValueError):
        comp.append(*steps[0])
    with pytest.raises(vec.VectorError) as e:
        vec.vector_append(sh, c, steps[0][0], steps[0][1], 0)
    assert e.value.status == -2


def _shifted(x):
    """The same rows, contiguous, one element into their storage."""
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    return y.copy_(x)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_append_rows_off_a_16_byte_boundary(dtype):
    U, d = 3, 64
    sh = vec.Shape(1, 1, U, U, d, vec.VECTOR_BF16 if dtype == torch.bfloat16 else vec.VECTOR_F32, 16)
    comp = Compressor(sh, vec.vector_plan_budget(200, 60, 10, 16), extra_rows=3)
    c, n = comp.cache, comp.cache.n_ret
    k, v = (torch.randn(U, d, device=DEV).to(dtype) for _ in range(2))
    for a, b in ((_shifted(k), v), (k, _shifted(v))):
        assert (a.data_ptr() | b.data_ptr()) % 16 and a.is_contiguous() and b.is_contiguous()
        comp.append(a, b, 5)
        assert torch.equal(c.ret_k[:, c.n_ret - 1], k) and torch.equal(c.ret_v[:, c.n_ret - 1], v)
        with pytest.raises(vec.VectorError) as e:
            vec.vector_append(sh, c, a, b, 5)
        assert e.value.status == -2
    assert c.n_ret == n + 2 and (c.ret_pos[:, n:n + 2] == 5).all()


def test_calls_go_to_the_current_stream():
    from paper_2605_23258_b200 import binding
    side = torch.cuda.Stream()
    for stream in (torch.cuda.current_stream(), side):
        with torch.cuda.stream(stream):
            assert binding._stream(None) == torch.cuda.current_stream().cuda_stream == stream.cuda_stream
