"""The share of exponentials on the FMA pipe is a build parameter that counts pairs: a share that the kernels would not run, and that
vector_score_exp2_fma_share would then report, does not compile."""
import subprocess

import pytest

from paper_2605_23258_b200 import build


@pytest.mark.parametrize("share,valid", [(4, True), (1, False), (5, False), (18, False)])
def test_only_whole_pairs_compile(tmp_path, share, valid):
    source = tmp_path / "share.cu"
    source.write_text('#include "score_tc.cuh"\nstatic_assert(vec::stc::POLY16 == %d);\n' % share)
    done = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, f"-DVECTOR_SCORE_POLY16={share}", "-c", str(source), "-o", str(tmp_path / "share.o")],
                          stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    assert (done.returncode == 0) == valid, done.stdout
    assert valid or "VECTOR_SCORE_POLY16" in done.stdout
