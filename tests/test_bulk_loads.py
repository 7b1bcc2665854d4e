"""The bulk loads of the kernels stay within the SM that issues them: the same library runs on one GPU and on the
ranks of several, where loads that deliver to a whole cluster are not used (CPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1312_1549_gb300", "csrc")


def test_no_bulk_load_delivers_to_a_cluster():
    loads = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for block in re.findall(r"asm(?:\s+volatile)?\s*\((.*?)\);", open(path).read(), flags=re.S):
            text = "".join(re.findall(r'"([^"]*)"', block))
            for instruction in text.split(";"):
                if "cp.async.bulk" in instruction:
                    loads += 1
                    assert "multicast" not in instruction, (os.path.basename(path), instruction)
    assert loads >= 2
