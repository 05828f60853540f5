"""Kernels that may start beside their predecessor read what it writes by plain
loads (no GPU): the read-only path (__ldg, or a load the compiler makes one of
for __restrict__ pointers) asks for memory that is constant over the kernel's
life and may be moved above the wait for the predecessor.  So in the sources it
reads only the plan's tables, which no kernel writes, and, in the zapping copy,
which is always a call's first kernel, the user's input."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1811_04165_gb300", "csrc")
# files -> the expressions read; `series` and `units` are the tables of the pre-sums' channels
TABLES = {
    "dedisperse_presum.cu": r"&a\.chunk_rows\[|&list\[|reinterpret_cast<const int4\*>\((units|series) \+",
    "dedisperse_step2.cu": r"&d2row0\[|&a\.d2\[",
    "snr.cu": r"a\.widths \+|widths \+ wi",
    "zap.cu": r"zap \+ c|reinterpret_cast<const uint4\*>\(row \+ p\)|row \+ p \+ b",
}


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_read_only_loads_are_of_tables():
    files = [f for ext in ("cu", "cuh", "h") for f in glob.glob(os.path.join(CSRC, f"*.{ext}"))]
    assert len(files) > 6
    for f in files:
        allowed = TABLES.get(os.path.basename(f), r"(?!)")
        reads = re.findall(r"__ldg\(([^;\n]*)", _code(f))
        other = [r for r in reads if not re.match(allowed, r)]
        assert not other, (os.path.basename(f), other)
        assert "ld.global.nc" not in _code(f)


def test_restrict_is_of_tables():
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        names = set(re.findall(r"__restrict__\s+(\w+)", _code(f)))
        # a batch's argument and work lists, written when the batch is made
        assert names <= {"passes", "work"}, (os.path.basename(f), names)
