"""Kernels that a dependent launch may start before their predecessor is done
(they call pdl_wait) read what it wrote: their arguments must not be declared
unchanging (`__restrict__` lets the compiler take the read-only path or move
a load above the wait), and nothing that a predecessor writes is read by
__ldg, which makes the same claim."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0709_3225_gb300", "csrc")
# set up once, before any launch
TABLES = ("thb", "centre", "centre2", "rep_of", "rep_of_cell", "cell0", "cw")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
            end = text.index("{", m.end())
            depth, k = 1, end + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            yield os.path.basename(path), m.group(1), text[m.end():end], text[end:k]


DEPENDENT = [(f, n, sig, body) for f, n, sig, body in _kernels() if "pdl_wait()" in body]


def test_there_are_some():
    assert len(DEPENDENT) >= 14


@pytest.mark.parametrize("file,name,sig,body", DEPENDENT, ids=[n for _, n, _, _ in DEPENDENT])
def test_arguments_may_change(file, name, sig, body):
    assert "__restrict__" not in sig
    for arg in re.findall(r"__ldg\(([^;]*)", body):
        assert any(re.search(rf"\b{t}\b", arg) for t in TABLES), arg


@pytest.mark.parametrize("file", ["lj_force_n3.cuh", "lj_slots.cuh", "lj_force_fx.cu", "lj_vjp_n3.cu", "lj_slots.cu", "lj_batch.cu"])
def test_counts_and_lists_are_plain_loads(file):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    for arg in re.findall(r"__ldg\(([^;]*)", text):
        assert not re.search(r"\b(cellq|onext|spos)\b", arg), arg
