"""Kernels launched overlapped run while the kernel before them may still be writing what they read after their wait: the
sources have no loads by the non-coherent path, and no `const __restrict__` inputs that let the compiler choose it."""
import os
import re

from paper_2410_01485_b200 import build

FORBIDDEN = [r"ld\.global\.nc", r"__ldg\s*\(", r"\bconst\s+[\w:]+\s*\*\s*(?:const\s+)?__restrict__",
             r"\b[\w:]+\s+const\s*\*\s*__restrict__"]


def test_no_non_coherent_loads():
    found = []
    for name in sorted(os.listdir(build.CSRC)):
        text = open(os.path.join(build.CSRC, name)).read()
        text = re.sub(r"//[^\n]*", "", text)
        found += [(name, m.group(0)) for pattern in FORBIDDEN for m in re.finditer(pattern, text)]
    assert found == []
