"""Dynamic shared memory that kernels read or fill 16 bytes at a time (uint4
rows, 16-byte asynchronous copies) is declared on 16 bytes: a kernel's own
shared arrays may come before it, so its start is only what it declares."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1110_1328_gb300", "csrc")
SIXTEEN = ("uint4", "ulonglong2")
# arrays of words that are read and written word by word
WORDS = {("allpairs.cu", "map"), ("band.cu", "s_rows"), ("verify.cu", "s_tab")}


def test_dynamic_shared_memory_starts_on_16_bytes():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        name, text = os.path.basename(path), open(path).read()
        for align, typ, var in re.findall(r"extern __shared__ (?:__align__\((\d+)\) )?([\w ]+?) (\w+)\[\]", text):
            seen += 1
            on16 = int(align or 0) >= 16 or typ in SIXTEEN
            assert on16 or (name, var) in WORDS, f"{name}: {var} is declared on less than 16 bytes"
    assert seen >= 8
