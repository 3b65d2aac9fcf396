"""Kernels that start before the launch ahead of them has ended (they call
pdl_wait) read fields by plain loads only. The non-coherent path is for memory
that nobody writes while the kernel lives, which holds for activity bytes, work
lists and coefficients, not for fields the launch ahead is still storing. Read
from the sources: a wrong load need not give a wrong value on any one run."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0901_1053_gb300", "csrc")
CONSTANT_LOADS = {"ld_word_if", "ld_mask2"}   # activity bytes


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def functions(text):
    """(name, body) of every device function and kernel."""
    for m in re.finditer(r"__(?:global|device)__[^;{]*?(?<!\w)(?!__launch_bounds__)(\w+)\s*\((?![^()]*\)\s+\w+\()", text):
        i = text.find("{", m.end())
        if i < 0 or text.find(";", m.end(), i) >= 0:   # a declaration
            continue
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        yield m.group(1), text[i:j]


ALL = {}
for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
    name = os.path.basename(path)
    for fn, body in functions(source(name)):
        ALL.setdefault(name, []).append((fn, body))


def reached(name):
    """The bodies of the overlapped kernels of a file and of the device
    functions they call, in it and in the shared quads."""
    fns = ALL[name] + (ALL["quads.cuh"] if "quads.cuh" in source(name) else [])
    todo = [(f, b) for f, b in fns if "pdl_wait()" in b]
    seen = {}
    while todo:
        f, b = todo.pop()
        if (f, b) in seen:
            continue
        seen[(f, b)] = True
        todo += [(g, c) for g, c in fns if g != f and re.search(r"\b%s\b" % g, b)]
    return list(seen)


FILES = [n for n in sorted(ALL) if any("pdl_wait()" in b for _, b in ALL[n])]


def test_every_overlapped_file_is_looked_at():
    assert {"kernels_band.cu", "kernels_half.cu", "kernels_slab.cu", "kernels_step.cu", "rz.cu"} <= set(FILES)
    assert "ldg_if" in [f for f, _ in reached("kernels_half.cu")]


@pytest.mark.parametrize("name", FILES)
def test_fields_are_read_by_plain_loads(name):
    for fn, body in reached(name):
        if re.search(r"ld\.global\.nc|__ldg", body):
            assert fn in CONSTANT_LOADS, (name, fn)
        for target in re.findall(r"__restrict__\s+\w+\s*=\s*(a\.\w+)", body):
            assert target not in ("a.in", "a.out"), (name, fn)
        for call in CONSTANT_LOADS:                    # and those loaders read activity bytes only
            for arg in re.findall(r"\b%s\(([^,()]*)" % call, body):
                assert not re.search(r"\b(a\.in|a\.out|in_of|out_of|in|out)\b", arg), (name, fn, arg)
