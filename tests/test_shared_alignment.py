"""Dynamic shared memory that a kernel fills in 16-byte words is declared with
that alignment."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_11449_gb300", "csrc")


def test_dynamic_shared_arrays_used_as_uint4_are_aligned():
    arrays = 0
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"extern __shared__ ([^;\[]+?)\s+(\w+)\[\]", text):
            arrays += 1
            scope = text[m.end():text.find("\n}\n", m.end())]
            if re.search(r"reinterpret_cast<(const )?uint4 \*>\(%s\b" % m.group(2), scope):
                assert m.group(1).endswith("uint4") or "__align__(16)" in m.group(1), f"{f}: {m.group(2)} is {m.group(1)}"
    assert arrays > 5
