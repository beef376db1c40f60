"""Every device allocation of the library can take the pooled scratch of the product entry points back:
none calls cudaMalloc but the helper that does."""
import glob
import os
import re

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2309_08572_gb300", "csrc")


def test_allocations_go_through_the_helper():
    calls = {}
    for path in glob.glob(os.path.join(CSRC, "*.c*")):
        with open(path) as f:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
        n = len(re.findall(r"\bcudaMalloc\s*\(", code))
        if n:
            calls[os.path.basename(path)] = n
    assert calls == {"tcgemm.cu": 2}      # the helper: before and after the pool is trimmed
