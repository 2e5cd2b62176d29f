"""Kernels that may start before the one in front of them has ended: after the wait
for it they read its results by plain loads.  A read-only load (__ldg) promises that
nobody writes the memory while the kernel runs, and may be moved before the wait."""
import os
import re

import pytest

from paper_1807_04638_gb300 import build


def source(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name,kernel,constant", [
    ("line.cuh", "k_line", ("tab",)),       # L and K over the band, written at creation
    ("plane.cuh", "k_spec_step", ()),
    ("stage.cuh", "k_stage2", ("get2(p)", "p", "p + dB")),  # the stored state
])
def test_read_only_loads_after_the_wait(name, kernel, constant):
    src = source(name)
    body = src[re.search(r"\b%s\(const __grid_constant__" % kernel, src).start():]
    body = body[:body.index("\n}\n")]
    before, wait, after = body.partition("after_previous();")
    assert wait, "the kernel waits for the one in front"
    reads = re.findall(r"\b(?:__ldg|ldg)\((?:\(const float[24]?\*\))?\(?([^;]*?)\)[;, )]", after)
    assert all(any(r.startswith(c) for c in constant) for r in reads), reads
