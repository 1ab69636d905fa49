"""The forms of the decode merge, on either side of each line of the rule between them, with RoPE records too and with units of so many
records that a lane reads two headers.  Sampled units against the oracle."""
import json
import os
import re
import subprocess
import sys

import pytest
import torch

import paper_2605_23258_b200 as vec

from helpers import decode_bound, decode_call, decode_errors, decode_problem

pytestmark = pytest.mark.gpu
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


def _checked(oracle, U, g, d, n_ret, n_apx, rope, mode=0):
    q, cache, W = decode_problem(U, g, d, torch.bfloat16, n_ret, n_apx, 71 + d + g)
    before = vec.vector_kernel_launches()
    out = decode_call(q, cache, W, rope, mode=mode)
    assert vec.vector_kernel_launches() - before == 2, "one launch: the merge was not reached"
    errs = decode_errors(oracle, q, cache, W, out, rope, sorted({0, 1, U // 2, U - 2, U - 1}))
    # rebuilt values are rounded to eleven bits: 2^-12 of a value each, and the sum of a head may cancel to a third
    assert errs.max() <= (8e-4 if mode == 1 else decode_bound(torch.bfloat16, d, rope)), errs.max()
    assert bool(torch.isfinite(out).all())


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("d,g,full", [(128, 1, 4), (128, 2, 4), (128, 2, 5), (128, 3, 2), (128, 3, 3), (128, 4, 2), (128, 4, 3), (64, 3, 4), (64, 4, 4), (64, 2, 8)])
def test_both_sides_of_a_line(oracle, d, g, full, rope):
    for U in (full * SMS, full * SMS + 1):
        _checked(oracle, U, g, d, 65, 70, rope)


@pytest.mark.parametrize("g,full", [(2, 4), (2, 6), (3, 3), (3, 4), (4, 3), (6, 1)])
def test_rebuilt_values(oracle, g, full):
    _checked(oracle, full * SMS, g, 128, 64, 130, False, mode=1)


# blocks of the streaming kernel a unit: 11 and 8.7 with three and four records each; beyond some 50 tiles a block the streaming form is taken
@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("U,g,d,n_ret,n_apx", [(13, 2, 128, 65536, 73728), (13, 4, 128, 65536, 73728), (17, 2, 64, 16384, 8192), (17, 4, 64, 16384, 8192), (17, 8, 64, 16384, 8192)])
def test_two_headers_a_lane(oracle, U, g, d, n_ret, n_apx, rope):
    _checked(oracle, U, g, d, n_ret, n_apx, rope)


def _merge_kernels(shapes):
    """The merge that each (d, g, U) takes, by its name in a profile: of a process of its own, since a process does not profile again and again."""
    program = """if True:
        import json, sys
        import torch
        from helpers import decode_call, decode_problem
        names = []
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            for d, g, U in json.loads(sys.argv[1]):
                decode_call(*decode_problem(U, g, d, torch.bfloat16, 64, 64, 5), False)
        print(json.dumps([e.name for e in sorted(prof.events(), key=lambda e: e.time_range.start) if "decode_merge" in e.name]))
    """
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(here), here, os.environ.get("PYTHONPATH", "")]))
    done = subprocess.run([sys.executable, "-c", program, json.dumps(shapes)], stdout=subprocess.PIPE, text=True, check=True, timeout=300, env=env)
    names = json.loads(done.stdout.splitlines()[-1])
    if not names:
        pytest.skip("no kernel names from the profiler")
    assert len(names) == len(shapes)
    return names


def test_many_units_keep_enough_in_flight():
    """Three blocks of 256 threads a multiprocessor took 28.6 us for 900 units of two heads and 96 rows, a thread a channel 25.3; two for
    384 units of four heads 16.3, three 14.7."""
    resident = {(128, 2, 3): 4, (128, 2, 5): 5, (128, 4, 2): 2, (128, 4, 3): 3, (64, 4, 5): 7}      # by units a multiprocessor
    names = _merge_kernels([(128, g, 6 * SMS + 12) for g in (1, 2, 3)] + [(d, g, full * SMS) for d, g, full in resident])
    assert all("decode_merge_channels" in name for name in names[:3]), names[:3]
    assert [re.search(r"decode_merge_bf16<.*?(\d+)\)?>", name).group(1) for name in names[3:]] == [str(r) for r in resident.values()]
