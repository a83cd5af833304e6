"""The static scratch size that the header states is the size that the source declares."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_noalloc_scratch_size():
    src = open(os.path.join(ROOT, "paper_2511_13894_gb300", "csrc", "kkt_eval.h")).read()
    k = {n: int(v) for n, v in re.findall(r"constexpr int (kEv\w+) = (\d+);", src)}
    doubles = (1 << 18) + (k["kEvRowQ"] + k["kEvColQ"]) * k["kEvBlocks"] + k["kEvOut"]
    hdr = open(os.path.join(ROOT, "include", "pdhgc.h")).read()
    stated = re.search(r"file-scope device array of ([\d,]+) bytes \(\(1 << 18\)\s*\*?\s*\+ (\d+) \* (\d+) \+ (\d+) doubles\)", hdr)
    assert stated, "the header states no size"
    size, q, blocks, extra = (int(v.replace(",", "")) for v in stated.groups())
    assert (q, blocks, extra) == (k["kEvRowQ"] + k["kEvColQ"], k["kEvBlocks"], k["kEvOut"])
    assert size == 8 * doubles
