"""Rules of the CUDA sources that no run shows broken."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2109_09965_gb300", "csrc")


def test_cycle_data_is_read_through_plain_pointers():
    """With programmatic launches a kernel starts before the one that writes
    its inputs has ended and waits inside (cgks_pdl.cuh); the compiler may
    treat loads through const __restrict__ pointers as invariant and move them
    above that wait.  Only mesh tables, which nothing writes while cycles run,
    and the arrays of the two copy kernels outside cycles are declared so."""
    tables = {"perm", "blk", "list", "ptab", "wenok"}
    outside = {"k_gather_state", "k_scatter_state"}
    seen = set()
    for path in glob.glob(os.path.join(CSRC, "cgks_*.cuh")):
        text = open(path).read()
        for m in re.finditer(r"(\w+)\(([^(){};]*__restrict__[^(){};]*)\)\s*\{", text):
            for name in re.findall(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", m.group(2)):
                seen.add(name)
                assert name in tables or m.group(1) in outside, (os.path.basename(path), m.group(1), name)
    assert tables - {"wenok"} <= seen
