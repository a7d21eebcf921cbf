"""Kernels that may begin before the one ahead of them on the stream has ended (launch_early) read
memory only after after_previous(), by loads that the compiler keeps behind it: not through __ldg,
ld.global.nc or const __restrict__ parameters, which promise that the memory does not change while
the kernel runs."""
import os
import re

import pytest

from paper_1908_09359_gb300 import build


def strip(text):
    return re.sub(r"//[^\n]*", "", text)


def early_files():
    names = [f for f in sorted(os.listdir(build.CSRC)) if f.endswith(".cu")]
    return [f for f in names if "after_previous()" in strip(open(os.path.join(build.CSRC, f)).read())]


def test_there_are_such_files():
    assert {"contract_f32.cu", "contract_tc.cu", "fused_env3.cu", "fused_f32.cu", "qr.cu"} <= set(early_files())


@pytest.mark.parametrize("name", early_files() + [f for f in sorted(os.listdir(build.CSRC)) if f.endswith(".cuh")])
def test_no_loads_that_may_move_ahead_of_the_wait(name):
    text = strip(open(os.path.join(build.CSRC, name)).read())
    assert "__ldg" not in text and "global.nc" not in text


@pytest.mark.parametrize("name", early_files())
def test_such_kernels_wait_first(name):
    text = strip(open(os.path.join(build.CSRC, name)).read())
    seen = 0
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\(([^{;]*)\)\s*\{", text):
        body = text[m.end():text.index("\n}\n", m.end())]
        if "after_previous()" not in body:
            # then it is launched the plain way only
            assert not re.search(r"launch_(early|chains)\(" + m.group(1) + r"\b", text), m.group(1)
            continue
        seen += 1
        assert "__restrict__" not in m.group(2), m.group(1)
        assert "return" not in body[:body.index("after_previous()")], m.group(1)
    assert seen
