"""The order between the two blocks of a pair, read from the sources: what one block writes to its shared memory for products that the
other issues is released and acquired at the scope of the cluster.  A barrier's arrivals and waits that name no scope order one block."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_23258_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_arrivals_at_another_block_release():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        lines = _source(name).splitlines()
        for i, line in enumerate(lines):
            if re.search(r"mbarrier\.arrive[\w.]*\.shared::cluster\.b64 _, ", line):
                found += 1
                assert ".cluster.shared::cluster" in line, (name, line.strip())
                assert ".release.cluster" in line or "fence.release.sync_restrict::shared::cta.cluster" in lines[i - 1], (name, line.strip())
    assert found == 1


def test_the_issuing_warp_acquires():
    text = _source("residual_layer_tc.cuh")
    warp = text[text.index("} else if (warp == LOADER_WARPS) {"):]
    warp = warp[:warp.index("mma_bf16")]
    for bar in ("acc_empty", "full"):
        wait = re.search(r"mbar_wait_warp(<CTAS>)?\(&sy\.%s\[" % bar, warp)
        assert wait and wait.group(1), bar
        assert "tma::acquire_pair<CTAS>();" in warp[wait.end():], bar
    assert re.search(r"mbar_test<CTAS>\(&sy\.full\[", warp) and warp.count("acquire_pair<CTAS>") == 2
