"""Order of the library's device work, read from its sources.

A caller's stream need not be ordered with the legacy default stream, so every launch and every
copy or clear of device memory names its stream.
"""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1004_5076_gb300", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            yield f, re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f), encoding="utf-8").read())


def test_every_launch_and_clear_names_its_stream():
    for f, src in _sources():
        assert not re.findall(r"\bcudaMemset\w*(?<!Async)\s*\(", src), f
        for args in re.findall(r"<<<(.*?)>>>", src, re.S):
            depth, commas = 0, 0
            for ch in args:
                depth += ch in "([{"
                depth -= ch in ")]}"
                commas += ch == "," and depth == 0
            assert commas == 3, (f, args)


def test_every_copy_names_its_stream():
    for f, src in _sources():
        assert not re.findall(r"\bcudaMemcpy\w*(?<!Async)\s*\(", src), f
