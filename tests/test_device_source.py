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


def _body(code, at):
    """The text from the first brace at or after `at` to its match."""
    i = j = code.index("{", at)
    depth = 0
    while True:
        depth += {"{": 1, "}": -1}.get(code[j], 0)
        j += 1
        if depth == 0:
            return code[i:j]


def _functions():
    """Bodies of every device function, by name (overloads together)."""
    out = {}
    for code in FILES.values():
        for m in re.finditer(r"__(?:global|device)__[^;{}]*?\b(\w+)\((?=[^;{}]*\{)", code):
            names = re.findall(r"(\w+)\(", code[m.start():code.index("{", m.start())])
            for name in names:
                out[name] = out.get(name, "") + _body(code, m.start())
    return out


def _launched_after():
    """Kernels launched with launch_after, also through a local variable."""
    out = set()
    for code in FILES.values():
        for m in re.finditer(r"launch_after\(([^,]*?),", code):
            arg = m.group(1)
            if "(*kern)" in arg:
                continue
            names = re.findall(r"\bk_\w+", arg)
            for var in [] if names else re.findall(r"\b[a-z]\w*", arg):
                for definition in re.findall(r"\b%s = ([^;]*);" % var, code):
                    names += re.findall(r"\bk_\w+", definition)
            assert names, arg
            out |= set(names)
    return sorted(out)


@pytest.mark.parametrize("kernel", _launched_after())
def test_kernels_launched_ahead_use_plain_loads(kernel):
    """A kernel launched ahead of its predecessor is resident while that one
    still writes.  Loads through the read-only path are defined only for data
    that nobody writes during a kernel's lifetime, so it must not have any,
    also not in the functions it calls; and it waits for its predecessor."""
    functions = _functions()
    todo, seen = [kernel], set()
    while todo:
        name = todo.pop()
        seen.add(name)
        for bad in ("__ldg", "__restrict__", "ld.global.nc", "__ldcs"):
            assert bad not in functions[name], (kernel, name, bad)
        todo += [f for f in set(re.findall(r"\b(\w+)(?:<[^;()]*>)?\(", functions[name])) if f in functions and f not in seen]
    assert "pdl_wait()" in functions[kernel]
    assert len(seen) > 1  # the calls were followed


def test_kernels_launched_ahead_are_found():
    assert {"k_gather", "k_colsum_umma", "k_row_bias", "k_decode_split", "k_decode_mma",
            "k_decode_combine"} <= set(_launched_after())


def test_order_behind_loads_before_the_wait():
    """The column sums read q and k before they wait for the row statistics,
    the only kernel to do so: those are launched in the ordinary way."""
    early = []
    for kernel in _launched_after():
        before = _functions()[kernel].split("pdl_wait()")[0]
        if re.search(r"tma_load|cp_async|bulk_g2s|load_q", before):
            early.append(kernel)
    assert early == ["k_colsum_umma"]
    assert "k_rowstats_umma" not in _launched_after()
