"""Instructions that need a warp's lanes together (PTX's .aligned forms) stand in
helpers that join the lanes with __syncwarp() first.  Their callers reach them
from loops whose lanes part (rows outside the grid, one issuing lane), where
nothing else makes the lanes meet again.  Read from the sources: without it the
result is undefined, and a run shows nothing as long as the compiler happens to
join them."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1104_1703_gb300", "csrc")


def _functions_with_aligned_asm():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        # helpers begin in the first column and end at the first brace there
        for m in re.finditer(r"^__device__[^;{]*?(\w+)\([^;{]*\)\s*\{(.*?)^\}|^__device__[^;{\n]*?(\w+)\([^;{\n]*\) \{(.*)\}$",
                             text, re.S | re.M):
            name, body = (m.group(1), m.group(2)) if m.group(1) else (m.group(3), m.group(4))
            if ".aligned" in body:
                yield os.path.basename(path), name, body


def test_every_aligned_instruction_follows_a_syncwarp():
    found = list(_functions_with_aligned_asm())
    names = {n for _, n, _ in found}
    assert {"tmem_alloc", "tmem_dealloc", "tmem_ld16", "cl_arrive", "cl_wait"} <= names
    total = sum(open(p).read().count(".aligned") for p in glob.glob(os.path.join(CSRC, "*.cu*")))
    # comments apart, every use stands in one of these helpers
    assert sum(b.count(".aligned") for _, _, b in found) == total - _in_comments()
    for path, name, body in found:
        assert 0 <= body.find("__syncwarp();") < body.find(".aligned"), (path, name)


def _in_comments():
    n = 0
    for p in glob.glob(os.path.join(CSRC, "*.cu*")):
        n += sum(c.count(".aligned") for c in re.findall(r"//.*", open(p).read()))
    return n
