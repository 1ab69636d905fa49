"""The order that programmatic dependent launches rest on, read from the sources: a kernel lets its dependents start
(griddepcontrol.launch_dependents) only directly behind its own griddepcontrol.wait.  Then all that came before a kernel's primary
has finished when it starts, whatever chain the calls form.  And what a kernel reads behind its wait is no read-only data to the
compiler, which could read that ahead of the wait."""
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


def _chain_files():
    """The sources that wait for a primary, and the headers that they include."""
    text = {os.path.basename(p): open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}
    files = {f for f in text if 'asm volatile("griddepcontrol.wait' in text[f]}
    while True:
        more = {h for f in files for h in re.findall(r'#include "(\w+\.cuh)"', text[f])} - files
        if not more:
            return {f: re.sub(r"//[^\n]*", "", text[f]) for f in files}
        files |= more


def test_nothing_read_behind_the_wait_is_read_only():
    files = _chain_files()
    assert len(files) >= 12 and "select.cuh" in files
    for name, text in files.items():
        assert not re.search(r"__ldg\b|\.nc\.", text), name
        starts = [m.start() for m in re.finditer(r"__global__|__device__", text)] + [len(text)]
        for lo, hi in zip(starts, starts[1:]):
            function = text[lo:hi]
            if re.search(r"const [\w:]+\s*\* __restrict__", function):        # only a kernel that is launched the ordinary way
                assert function.startswith("__global__") and "griddepcontrol" not in function and "_role<" not in function, \
                    (name, function[:120])


def test_routing_reads_nothing_ahead_of_the_wait():
    """Every list that a routing kernel reads was written by a kernel of its chain: ahead of its wait it does not so much as name one."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "route.cu")).read())
    kernels = 0
    for m in re.finditer(r"__global__[^{;]*?(\w+)\(([^(){;]*)\) \{(.*?)\n\}", text, re.S):
        ahead, wait, _ = m.group(3).partition('asm volatile("griddepcontrol.wait')
        inputs = re.findall(r"const [\w:]+\* (?:__restrict__ )?(\w+)", m.group(2))
        if wait:
            kernels += 1
            assert inputs and not re.search(r"\b(%s)\b" % "|".join(inputs), ahead), (m.group(1), inputs)
    assert kernels == 5
