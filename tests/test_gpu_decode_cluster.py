"""Decode of few units in one launch (a thread block cluster per unit) against the oracle: cluster sizes from two to
sixteen, more blocks than heads and the other way round, blocks whose warps get no tile, and the neighbouring sizes that
take the two-kernel form.  The first and last rows of the pools and those at tile edges carry visible shares of the output
(helpers.decode_problem); tolerances: helpers.decode_bound, and 2^-8 more for a bf16 output."""
import pytest
import torch

from helpers import decode_bound, decode_call, decode_errors, decode_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("d,U,g,n_ret,n_apx", [
    (128, 1, 8, 65, 0),            # two tiles: a cluster of two, each with one tile
    (128, 3, 1, 700, 1100),        # more blocks than heads
    (128, 17, 8, 129, 300),        # five tiles
    (128, 37, 4, 500, 900),        # clusters of a few blocks
    (128, 74, 3, 100, 200),        # four tiles, at most two blocks a unit
    (128, 75, 2, 100, 200),        # one unit more than that
    (64, 5, 6, 1000, 2500),
    (64, 2, 2, 0, 129),            # key-only tiles alone
])
def test_decode_cluster(oracle, rope, d, U, g, n_ret, n_apx):
    q, cache, W = decode_problem(U, g, d, torch.bfloat16, n_ret, n_apx, U * 100 + g, sharp=2.0)
    units = range(0, U, max(1, U // 4))
    bound = decode_bound(torch.bfloat16, d, rope)
    for out_dtype, more in ((torch.float32, 0.0), (torch.bfloat16, 2.0 ** -8)):
        errs = decode_errors(oracle, q, cache, W, decode_call(q, cache, W, rope, out_dtype), rope, units)
        assert errs.max() <= bound + more, errs.max()
