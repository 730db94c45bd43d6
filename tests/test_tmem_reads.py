"""Every TMEM read in the sources waits within its own statement (CPU).  The
registers of a tcgen05.ld hold nothing until tcgen05.wait::ld; between two
statements a compiler may move or spill them, and the kernel would compute
with what was there before."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15171_gb300", "csrc")


def test_a_read_and_its_wait_are_one_statement():
    reads = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path, encoding="utf-8") as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for asm in re.findall(r"\basm\b.*?\)\s*;", text, re.S):
            if "tcgen05.ld." in asm:
                reads += 1
                assert asm.rindex("tcgen05.ld.") < asm.find("tcgen05.wait::ld"), f"{os.path.basename(path)}: {asm[:80]}"
    assert reads >= 3
