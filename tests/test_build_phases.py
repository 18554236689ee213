"""The one-pass build's warps share a vector in shared memory: tokens are set in
any of its words by any lane, each lane reads and clears words of its own.  A
race between the two shows only when a warp's lanes run apart, which no run can
be made to do, so the order of the phases is checked in the source."""
import re

from tests.conftest import ROOT


def test_one_pass_build_fences_its_vector():
    src = (ROOT / "paper_1708_04329_gb300" / "csrc" / "grim_build.cu").read_text()
    start = src.index("for (uint32_t c = 0; c <= 32 + a.k;")
    body = src[start:src.index("if (!ROWS ||", start)]
    found = re.findall(r"set_tokens\(|v\[w \* 32 \+ lane\]|__syncwarp\(\)", body)
    assert found.count("set_tokens(") == 2 and found.count("v[w * 32 + lane]") == 3
    last = None  # the kind of access since the last fence
    for x in found * 2:  # the loop's end meets its start
        if x == "__syncwarp()":
            last = None
            continue
        assert last in (None, x), "lanes' own words and any lane's words without a fence between"
        last = x
