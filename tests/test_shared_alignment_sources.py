"""Shared arrays that kernels write or read as 8- or 16-byte packs are declared
with that alignment: a static array has only its element type's otherwise, and
a pack at another address is a misaligned access."""
import os
import re

from paper_1512_03662_gb300 import build


def test_packed_shared_arrays_are_aligned():
    found = 0
    for name in build.SOURCES:
        with open(os.path.join(build.CSRC, name)) as f:
            s = re.sub(r"//[^\n]*", "", f.read())
        packed = set(re.findall(r"(?:load|store)_pack<[^>]*>\(\s*&(\w+)\[", s))
        for line in re.findall(r"[^\n;]*__shared__[^;]*;", s):
            for array in re.findall(r"(\w+)\[", line):
                if array in packed:
                    found += 1
                    assert "__align__(16)" in line, (name, line.strip())
    assert found == 1
