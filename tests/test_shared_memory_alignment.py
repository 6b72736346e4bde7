"""A dynamic shared array that holds fixed-point limbs is read in 16-byte
vectors, so its declaration states that alignment (the type alone, double,
promises 8 bytes)."""
import glob
import os
import re

from paper_1601_06681_gb300 import build


def dynamic_shared_arrays():
    """(file, alignment stated, declared name, the function's body) of each declaration."""
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu"))):
        src = open(path).read()
        for m in re.finditer(r"extern __shared__ (?:__align__\((\d+)\) )?[\w ]+ (\w+)\[\];", src):
            body = src[m.end():src.index("\n}\n", m.end())]
            yield os.path.basename(path), int(m.group(1) or 0), m.group(2), body


def test_arrays_of_limbs_are_declared_16_byte_aligned():
    found = [(f, a, n) for f, a, n, body in dynamic_shared_arrays()
             if re.search(r"reinterpret_cast<(?:int2|int4|uint4)\*>\(%s\)" % n, body)]
    assert len(found) >= 5
    assert [v for v in found if v[1] < 16] == []
