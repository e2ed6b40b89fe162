"""Kernels whose launch overlaps the previous kernel (launch_next, launch_after), as
the sources state them: each waits for that kernel first, and none promises that
its inputs are constant for the whole kernel.  A const pointer that is
__restrict__ as a kernel parameter lets the compiler read it before the wait,
while the kernel before may still be writing."""

import glob
import os
import re

WAITS = ("after_previous();", "wait_previous();")
CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2401_02756_gb300", "csrc")


def _balanced(text, at):
    """text[at] is '(': the index past its ')'."""
    depth = 0
    for i in range(at, len(text)):
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced")


def _kernels():
    """{name: (parameters, start of the body)} of every __global__ function."""
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__\s+void\s+", text):
            rest = text[m.end():]
            bounds = re.match(r"__launch_bounds__\s*", rest)
            if bounds:
                rest = rest[_balanced(rest, bounds.end()):]
            name = re.match(r"\s*(\w+)\s*\(", rest)
            end = _balanced(rest, name.end() - 1)
            body = rest[end:].lstrip()
            if body.startswith("{"):  # (a definition)
                out[name.group(1)] = (rest[name.end():end - 1], body[1:].lstrip())
    return out


def _overlapped():
    names = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"launch_(?:next\(\s*[^,()]+,|after\()\s*(\w+)", text):
            names.add(m.group(1))
        for m in re.finditer(r"auto kern = ([^;]*);", text):  # (a kernel named through a variable)
            if "launch_next(overlap, kern" in text or "launch_after(kern" in text:
                names.update(re.findall(r"\bk_\w+", m.group(1)))
    return {n for n in names if n.startswith("k_")}


def test_every_overlapped_kernel_waits_first():
    kernels = _kernels()
    names = _overlapped()
    assert len(names) > 25 and names <= set(kernels)
    late = [n for n in names if not kernels[n][1].startswith(WAITS)]
    assert not late, late


def test_no_restrict_parameter_where_the_launch_overlaps():
    promised = [n for n, (params, body) in _kernels().items()
                if body.startswith(WAITS) and "__restrict__" in params]
    assert not promised, promised
