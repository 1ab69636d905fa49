"""The order that programmatic dependent launches rest on, read from the sources: a kernel lets its dependents start
(griddepcontrol.launch_dependents) only directly behind its own griddepcontrol.wait.  Then all that came before a kernel's primary
has finished when it starts, whatever chain the calls form."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_23258_b200", "csrc")


def test_dependents_start_behind_the_wait():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        lines = [line for line in open(path).read().splitlines() if not line.strip().startswith("//")]
        for i, line in enumerate(lines):
            if re.search(r'asm volatile\("griddepcontrol\.launch_dependents', line):
                found += 1
                assert re.match(r'\s*asm volatile\("griddepcontrol\.wait', lines[i - 1]), f"{os.path.basename(path)}: {line.strip()}"
    assert found >= 15
