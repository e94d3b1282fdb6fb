"""Kernels raise the bits of the control block's error word with atomicOr alone: other
CTAs of the same launch may be raising another bit of it, or polling one as their
signal to give up, and a plain read-modify-write can undo what they raised."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_04838_gb300", "csrc")


def test_error_bits_are_raised_atomically():
    atomic = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            for n, line in enumerate(f, 1):
                code = line.split("//")[0]
                assert not re.search(r"(->|\.)err\s*([|&^+-]?=)(?!=)", code), "%s:%d: %s" % (name, n, line.strip())
                atomic += len(re.findall(r"atomicOr\(&[^;]*err, [124]\)", code))
    assert atomic >= 4
