"""Dynamic shared memory starts where its declaration's alignment lets it, behind the
kernel's static shared variables: an array that a kernel reads as anything wider than its
declared elements has to ask for the alignment itself (CPU, from the source text)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_10982_gb300", "csrc")
SIZE = {"unsigned char": 1, "uint16_t": 2, "int32_t": 4, "uint32_t": 4, "float": 4, "int64_t": 8, "unsigned long long": 8}
DECL = re.compile(r"extern __shared__ (__align__\((\d+)\) )?([\w ]+?) (\w+)\[\];")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))), ids=os.path.basename)
def test_widened_arrays_ask_for_their_alignment(path):
    text = open(path).read()
    for m in DECL.finditer(text):
        align, element, name = int(m.group(2) or 0), m.group(3), m.group(4)
        # casts of a pointer into the array: to a type of known size, or one that may be of any (16)
        casts = [SIZE.get(c.strip(), 16) for c in re.findall(r"reinterpret_cast<(?:const )?([\w ]+?) ?[*&]>\(" + name + r"\b", text)]
        # produce() lays 16-byte records out behind the keys it is handed
        widest = max(casts + [SIZE[element]] + [16] * (name == "key" and "reinterpret_cast<uint4 *>(rest)" in text))
        assert widest <= max(align, SIZE[element]), f"{os.path.basename(path)}: {m.group(0)} is read {widest} bytes at a time"
