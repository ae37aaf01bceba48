"""Kernels that may be resident while their inputs are still written (they call
dependent_begin) read through the coherent path: the read-only path wants data
that nobody writes while the kernel lives, and griddepcontrol.wait says nothing
about it.  The rule is checked on the sources: every file that holds such a
kernel, or device code that one of them calls."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_03732_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg\s*\(|ld\.global\.nc|tex1Dfetch")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels(text):
    """(parameters, body) of every kernel of a source file."""
    for k in re.finditer(r"__global__[^;{]*?\bk_\w+\(([^)]*)\)\s*\{", text):
        depth, end = 1, k.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        yield k.group(1), text[k.end():end]


@pytest.mark.parametrize("name", ["rlt2_ascent.cuh", "rlt2_lap.cuh", "rlt2_movefx.cuh"])
def test_shared_device_code_reads_coherently(name):
    assert not READ_ONLY.search(_code(name))


def test_dependent_kernels_read_coherently():
    found = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        text = _code(name)
        dependent = [k for k in _kernels(text) if "dependent_begin()" in k[1]]
        found += len(dependent)
        for params, body in dependent:
            assert "__restrict__" not in params and not READ_ONLY.search(body), name
        if dependent:  # its device functions may be called from them
            assert not READ_ONLY.search(text), name
    assert found >= 6
