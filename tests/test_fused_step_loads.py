"""The one-launch 2D step reads what the launch before it writes by ordinary loads
(csrc/step2d_fused.cu, read as text).

Its launches are programmatic dependent ones, so a launch may start while the one
that writes phi, u* and the populations still runs.  __ldg and loads that the
compiler may make read-only (through const __restrict__ parameters) are defined only
for data that nobody writes during the kernel, and need not stay behind the wait for
the launch before."""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_0902_3921_gb300", "csrc", "step2d_fused.cu")


def test_ordinary_loads_after_the_wait():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    start = text.index("step2d_kernel(const float")
    kernel = text[start:text.index("\ntemplate", start)]
    assert "__ldg" not in kernel and "ld.global.nc" not in kernel
    assert "__restrict__" not in kernel[:kernel.index("{")]
    # no global load is written before the wait: the lambdas that load are called behind it
    before = kernel[kernel.index("{"):kernel.index("pdl_wait()")]
    for name in re.findall(r"auto (\w+) = \[&\]", before):
        assert not re.search(rf"(?<!auto )\b{name}\(", before) or name in ("rowof",), name
