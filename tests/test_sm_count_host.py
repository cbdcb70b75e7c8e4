"""The number of SMs stands in one place: the lines between kernel forms and
block sizes are counted in tiles an SM, and two copies of one line that must
agree cannot drift apart."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_31481_gb300", "csrc")


def test_the_sm_count_is_named_once():
    found = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh", ".cpp", ".h")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
        found += [f"{f}: {m.group(0).strip()}" for m in re.finditer(r"[^\n]*\b(?:76|152|304)\b[^\n]*", code)]
    assert found == ["fst_layout.h: constexpr int kSms = 152;"], found
