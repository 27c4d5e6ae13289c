"""Dynamic shared memory is declared with the alignment its accesses need.

The projector kernels read structures of 16-byte alignment (float4 tables, view
parameters) from it.  A declaration without an alignment promises one byte only:
behind static shared data that is no multiple of 16 bytes (the persistent back
projection has 4104 bytes), a 16-byte access could then be misaligned.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_03172_gb300", "csrc")


def _declarations():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            for number, line in enumerate(f, 1):
                code = line.split("//")[0]
                if re.search(r"\bextern\b.*\b__shared__\b|\b__shared__\b.*\bextern\b", code):
                    yield f"{name}:{number}", code


def test_there_are_declarations():
    assert len(list(_declarations())) >= 6


@pytest.mark.parametrize("where,code", list(_declarations()))
def test_dynamic_shared_memory_is_aligned(where, code):
    m = re.search(r"__align__\((\d+)\)|alignas\((\d+)\)", code)
    assert m and int(m.group(1) or m.group(2)) % 16 == 0, f"{where}: {code.strip()}"
