"""Properties of the device sources that no run can show reliably."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_3339_gb300", "csrc")


def test_every_tensor_memory_load_waits_in_its_own_statement():
    # tcgen05.ld is asynchronous: its registers may be read only after tcgen05.wait::ld, and only one
    # asm statement holding both keeps the compiler's arithmetic on them behind the wait
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for stmt in re.findall(r"\basm\b.*?\)\s*;", src, flags=re.S):
            if "tcgen05.ld." in stmt:
                found += 1
                assert stmt.find("tcgen05.wait::ld") > stmt.find("tcgen05.ld."), os.path.basename(path) + ": " + stmt
    assert found >= 3
