"""Dynamic shared memory that kernels read 16 bytes at a time is declared with that alignment: beside a static shared variable
nothing else places it on such a boundary."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_17132_gb300", "csrc")
WIDE = re.compile(r"\b(float4|double2|uint4|cp_async16|cp_async_elem)\b")


def test_files_with_wide_shared_accesses_declare_the_alignment():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        if not WIDE.search(text):
            continue
        for line in re.findall(r"extern __shared__[^;]*;", text):
            if " double " in line:  # read element by element
                continue
            seen += 1
            assert "__align__(16)" in line, (name, line)
    assert seen >= 5
