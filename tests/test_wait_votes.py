"""Bounded waits of whole warps are decided for the whole warp: in the kernels whose roles run
warp-wide instructions after a wait (tcgen05.ld, __syncwarp), a wait decided lane by lane is left
to one elected thread, or its result is not used.  What a kernel waits for before it ends (its
copies and its MMAs) is waited for whatever the error flag says."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2501_07047_gb300" / "csrc"
ELECTED = re.compile(r"if \((lane|tid|threadIdx\.x) == 0")


def per_lane_decisions(source):
    """Line numbers of tc::mbar_wait calls whose result decides something outside the block of an
    elected thread."""
    found, blocks, head = [], [], ""
    for number, line in enumerate(source.splitlines(), 1):
        code = line.split("//")[0]
        if "tc::mbar_wait(" in code and not code.strip().startswith("tc::mbar_wait("):
            if not any(ELECTED.search(b) for b in blocks) and not ELECTED.search(code):
                found.append(number)
        for ch in code:
            if ch == "{":
                blocks.append(head)
                head = ""
            elif ch == "}":
                blocks.pop()
                head = ""
            elif ch == ";":
                head = ""
            else:
                head += ch
    return found


def test_the_scan_sees_a_decision_by_lanes():
    planted = "void k() {\n  if (lane == 0) {\n    if (!tc::mbar_wait(b)) return;\n  }\n  if (!tc::mbar_wait(b)) return;\n}\n"
    assert per_lane_decisions(planted) == [5]


@pytest.mark.parametrize("name", ["bconv_tc.cu", "bconv_cc_tma.cu", "ntt_tc.cu", "ntt_tc2.cu"])
def test_warps_decide_together(name):
    assert per_lane_decisions((CSRC / name).read_text()) == []


@pytest.mark.parametrize("name", ["bconv_tc.cu", "bconv_cc_tma.cu", "ntt_tc.cu", "ntt_tc2.cu"])
def test_last_waits_ignore_the_error_flag(name):
    """tc::mbar_wait gives up as soon as another thread has; a wait whose result nobody uses is such a
    last one and takes tc::mbar_drain."""
    code = [line.split("//")[0].strip() for line in (CSRC / name).read_text().splitlines()]
    assert [c for c in code if re.search(r"(^|\bif \(\w+\[\w+\]\) )tc::mbar_wait\(", c)] == []
    assert any("tc::mbar_drain(" in c for c in code)
