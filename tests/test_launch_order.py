"""Kernels launched before the kernels ahead of them in the stream have ended
(programmatic launches, recognised by their wait) make no promise that the
memory they read does not change while they run: no __restrict__ on their
pointers or on those of the bodies they inline, no __ldg.  Either lets the
compiler read ahead of the wait, or through the read-only path."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1105_5804_gb300", "csrc")


def _code(path):
    src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", src)


def _kernels(src):
    """(name, parameters and body) of every __global__ function."""
    for m in re.finditer(r"__global__", src):
        start = src.index("{", m.end())
        depth, i = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
            if depth == 0:
                break
        head = src[m.end():start]
        yield re.findall(r"\b(k\w*)\s*\(", head)[0], head + src[start:i]


FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_read_only_promise(path):
    src = _code(path)
    assert "__ldg(" not in src
    if path.endswith(".cuh"):
        assert "__restrict__" not in src
    for name, text in _kernels(src):
        if "wait_for_previous()" in text:
            assert "__restrict__" not in text, name
            body = text[text.index("{") + 1:]
            called = set(re.findall(r"\b(\w+)\s*(?:<[^;{}()]*>)?\(", body))
            for f in called:   # device functions of the same file
                m = re.search(r"__device__ __forceinline__ [\w&* ]*\b%s\(([^{]*)\{" % f, src)
                assert not (m and "__restrict__" in m.group(1)), (name, f)


def test_the_programmatic_kernels_are_found():
    names = [n for p in FILES for n, text in _kernels(_code(p)) if "wait_for_previous()" in text]
    assert len(names) >= 20 and {"k_sw_label", "k_merge", "k3_local", "k_pixel_bonds", "k_sw_small"} <= set(names)
