"""Every wait inside a kernel is bounded and ends in an abort that all of a
block's warps follow.  A warp that issues tensor-core products as a whole
(elect.sync over all 32 lanes) must not lose a lane between them: it has no way
out of its loops but on an outcome that its lanes agreed on.  Read from the sources, since a wait
that runs out there cannot be staged short of a kernel that stalls."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_03395_gb300", "csrc")


@pytest.mark.parametrize("name,sections", [("ffx_planes.cu", 3), ("ffx_tc16.cu", 2)])
def test_product_warps_leave_as_one(name, sections):
    with open(os.path.join(CSRC, name)) as f:
        source = f.read()
    found = re.findall(r"// -+ products: the whole warp.*?(?=// -+ epilogue)", source, re.S)
    assert len(found) == sections
    for body in found:
        assert not re.search(r"\b(break|return|continue);", body)
        # a loop that may end early tests an outcome the lanes agreed on
        early = re.findall(r"for \([^;]*; (\w+) &&", body)
        assert all(f"{flag} = __all_sync(0xffffffffu, {flag});" in body for flag in early)
