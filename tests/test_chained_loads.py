"""Kernels of chained launches read nothing that a kernel before them writes as
data that stays unchanged: the next kernel of a chain is resident while the one
before still writes the state, so the read-only loads (ld.global.nc, __ldg, and
those that the compiler makes from __restrict__) are for the masks alone."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1206_0389_gb300", "csrc")


def code(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"/\*.*?\*/", "", f.read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def test_the_list_below_holds_every_file_of_chained_kernels():
    users = {f for f in os.listdir(CSRC) if f != "chained.cuh" and "begin_chained()" in code(f)}
    assert users == {"update.cuh", "adjoint.cu"}


@pytest.mark.parametrize("name", ["update.cuh", "adjoint.cu"])
def test_state_is_read_by_coherent_loads(name):
    text = code(name)
    assert ".nc" not in text and "__restrict__" not in text
    assert all(arg.startswith("a.masks") for arg in re.findall(r"__ldg\(([^)]*)", text))
    # the decode of Store reads through __ldg (kernels that are never chained use it)
    assert "::template get" not in text
    for asm in re.findall(r"asm[^;]*?\(\"ld\.[^;]*;[^;]*;", text):
        assert asm.startswith("asm volatile") and '"memory"' in asm, asm
