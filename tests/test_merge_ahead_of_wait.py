"""What the decode merge may touch ahead of its wait for the streaming kernel, read from the source: the map, which that kernel does not
write, and nothing that it does."""
import os
import re

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_23258_b200", "csrc", "decode_bf16.cuh")


def _kernels():
    text = re.sub(r"//[^\n]*", "", open(HEADER).read())
    return {m.group(1): (m.group(2), m.group(3)) for m in re.finditer(r"__global__[^{;]*?(decode_merge_\w+)\(([^(){;]*)\) \{(.*?)\n\}", text, re.S)}


def test_only_the_map_is_read_ahead_of_the_wait():
    kernels = _kernels()
    assert set(kernels) == {"decode_merge_bf16", "decode_merge_channels"}
    for name, (args, body) in kernels.items():
        ahead, wait, behind = body.partition('asm volatile("griddepcontrol.wait')
        assert wait and "partial" in args and "out" in args
        assert not re.search(r"\b(partial|out)\b", ahead), name
        assert re.search(r"\bpartial\b", behind) and re.search(r"\bout\b", behind), name
        # a pointer that is named ahead of the wait leads to the map
        assert set(re.findall(r"\*\s*(?:__restrict__ )?(\w+)(?=,|\)|$)", args)) & set(re.findall(r"\w+", ahead)) <= {"W"}, name
