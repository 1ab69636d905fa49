"""Streaming decode under RoPE decoupling against the oracle, more units than the one-launch form takes: key-only tiles that
end in their first or second half, units that begin and end inside a block, teams that meet no key-only tile or no tile at
all, one to eight heads.  The first and last rows of the pools and those at tile edges carry visible shares of the output
(helpers.decode_problem); tolerances: helpers.decode_bound."""
import pytest
import torch

from helpers import decode_bound, decode_call, decode_errors, decode_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("U,g,n_ret,n_apx", [
    (75, 1, 1, 1),                 # two tiles a unit, one row each
    (80, 8, 70, 1000),             # eight key-only tiles, the last of 104 rows
    (150, 4, 300, 0),              # retained tiles alone
    (90, 3, 0, 321),               # key-only tiles alone, the last of 65 rows: one row in its second half
    (76, 5, 640, 6400),            # buffers and slots used over and over
])
def test_decode_stream_rope(oracle, d, U, g, n_ret, n_apx):
    q, cache, W = decode_problem(U, g, d, torch.bfloat16, n_ret, n_apx, U * 10 + g, sharp=2.0)
    out = decode_call(q, cache, W, True, times=2)      # the second call meets the records of the first
    errs = decode_errors(oracle, q, cache, W, out, True, sorted({0, 1, U // 2, U - 2, U - 1}))
    assert errs.max() <= decode_bound(torch.bfloat16, d, True), errs.max()
