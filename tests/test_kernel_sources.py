"""What holds for kernels that come in while the launch before them still runs (griddepcontrol.wait), checked on their
source: the wavefields, which that launch writes, are read by ordinary loads through plain pointers.  A read-only load
(__ldg, ldg4, a const __restrict__ pointer) may be moved before the wait or be served from a cache that was filled
before it, and no test of the results could be relied on to show it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_02362_gb300", "csrc")
EARLY = [p for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))) if "griddepcontrol.wait" in open(p).read()]
# the fields of the arguments that no launch in flight writes: model, sponge tables, receivers and their data
CONSTANT = r"a\.(c|gx|gz|inj_next|inj_map)\b|val \+"


def test_there_are_such_kernels():
    assert [os.path.basename(p) for p in EARLY] == ["fwime_prop.cuh", "k_pair.cu"]


@pytest.mark.parametrize("path", EARLY, ids=os.path.basename)
def test_wavefields_are_read_plainly(path):
    src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    assert "__restrict__" not in src
    src = src.replace("float4 ldg4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }", "")
    loads = re.findall(r"(?:__ldg|ldg4|__ldca|__ldcg)\(([^;]*)", src)
    assert loads
    for arg in loads:
        assert re.match(CONSTANT, arg), arg[:60]
