"""The merge of the streaming decode: blocks that merge a range of the units, ordered by map (several sequences share one, a range ends
within a map's sequences or passes into the next map's), a block a unit with more than four heads, and units of so many records that a
lane reads two headers.  Sampled units against the oracle; with no retained or no key-only rows too."""
import numpy as np
import pytest
import torch

import paper_2605_23258_b200 as vec

from helpers import decode_bound, decode_errors, decode_problem

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _decode(q, cache, W, batch, mode, out_dtype):
    U, g, d = q.shape
    LH = U // batch
    sh = vec.Shape(batch, 1, LH * g, LH, d, vec.VECTOR_BF16, 16, 7)
    out = torch.full(q.shape, float("nan"), dtype=out_dtype, device=DEV)
    ws = vec.alloc_workspace(sh, vec.vector_plan_budget(16384, 8192, -1, 16))
    vec.vector_decode_attn(sh, q, cache, W, out, mode, ws)
    torch.cuda.synchronize()
    assert vec.vector_device_fault() == 0
    return out


@pytest.mark.parametrize("d,g,batch,maps,n_ret,n_apx,mode", [
    (128, 4, 5, 120, 70, 200, 0), (128, 3, 1, 297, 65, 0, 0), (128, 1, 7, 70, 130, 129, 0), (128, 2, 445, 1, 0, 90, 0), (128, 8, 3, 150, 64, 300, 0),
    (128, 5, 100, 1, 64, 128, 0), (64, 2, 9, 140, 70, 200, 0), (64, 1, 2, 600, 65, 1, 0), (64, 4, 2, 300, 64, 300, 0), (64, 7, 4, 90, 100, 300, 0),
    (128, 4, 1, 13, 16384, 8192, 0), (128, 8, 1, 13, 16384, 8192, 0), (128, 4, 5, 120, 70, 200, 1), (128, 6, 3, 40, 70, 200, 1)])
def test_decode_merge(oracle, d, g, batch, maps, n_ret, n_apx, mode):
    U = batch * maps
    q, cache, W = decode_problem(U, g, d, torch.bfloat16, n_ret, n_apx, 53 + d + g)
    W = W[:maps].contiguous()
    out = _decode(q, cache, W, batch, mode, torch.float32)
    units = sorted({0, 1, 2, maps - 1, min(maps, U - 1), U // 2, U - 2, U - 1} & set(range(U)))
    errs = decode_errors(oracle, q, cache, W.repeat(batch, 1, 1), out, False, units)
    # rebuilt values are rounded to eleven bits: 2^-12 of a value each, and the sum of a head may cancel to a third
    assert errs.max() <= (8e-4 if mode == 1 else decode_bound(torch.bfloat16, d, False)), errs.max()
    assert torch.equal(_decode(q, cache, W, batch, mode, torch.bfloat16), out.to(torch.bfloat16))
    # every unit: a sequence gives bit for bit what it gives when its map is its own
    if mode == 0 and batch > 1:
        alone = _decode(q, cache, W.repeat(batch, 1, 1).contiguous(), 1, mode, torch.float32)
        assert torch.equal(alone, out)
    assert np.isfinite(out.cpu().numpy()).all()
