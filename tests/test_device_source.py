"""Properties of the CUDA sources that no run shows while the toolchain is kind."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_00188_gb300", "csrc")


def _code(path):
    """The file without its comments."""
    with open(path) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


FILES = {os.path.basename(p): _code(p) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


@pytest.mark.parametrize("name", [f for f in FILES if "extern __shared__" in FILES[f]])
def test_dynamic_shared_memory_aligned_by_type(name):
    """Dynamic shared memory follows a kernel's static shared memory, at the
    alignment of the declared type and no more.  A kernel reads it 16 bytes at
    a time, so the type carries that alignment, unless the kernel takes raw
    bytes and rounds the base up itself."""
    found = re.findall(r"extern __shared__ ([\w ()]+?) (\w+)\[\];([^;]*;)", FILES[name])
    assert found
    for kind, var, following in found:
        own = kind == "uint8_t" and re.search(r"align1024\(%s\)|%s \+ \(\(1024u" % (var, var), following)
        assert own or kind in ("float4", "uint4"), (name, kind, var)
