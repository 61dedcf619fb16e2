"""Shared-memory arrays that a kernel accesses through a wider vector type declare its
alignment (an array has only that of its element type otherwise)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1612_01287_gb300", "csrc")
ALIGN = {"unsigned char": 1, "float": 4, "int": 4, "float2": 8, "double": 8, "uint64_t": 8,
         "float4": 16, "double2": 16, "int4": 16, "uint4": 16}
DECL = re.compile(r"__shared__\s+(?:__align__\((\d+)\)\s+)?([a-z][\w ]*?)\s+(\w+)\s*\[")


def test_vector_accesses_are_aligned():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(path).read()
        for m in DECL.finditer(text):
            align = max(int(m.group(1) or 1), ALIGN[m.group(2)])
            body = text[m.end():].split("__global__")[0]  # the rest of the kernel
            for t in re.findall(r"reinterpret_cast<(?:const )?(\w+)\*>\(&?%s\b" % m.group(3), body):
                seen += 1
                assert align >= ALIGN.get(t, 1), (os.path.basename(path), m.group(0), t)
    assert seen > 0
