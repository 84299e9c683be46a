"""A kernel's limit of dynamic shared memory belongs to every host thread, so no
launch sets it to its own need (a launch on another thread would find it
lowered): on the sources, each setting is a constant of the kernel, or all that
the device has (smem_limit)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_07537_gb300", "csrc")


def settings(text):
    """The size expressions of every setting of the limit."""
    for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize\s*,", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield " ".join(text[m.end():i - 1].split())


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_limits_are_constants(name):
    for size in settings(open(os.path.join(CSRC, name)).read()):
        if size == "(int)((size_t)most - fa.sharedSizeBytes)":  # smem_limit
            assert name == "common.cuh"
            continue
        left = re.sub(r"\(int\)|sizeof\(\w+\)|\bk[A-Z]\w*|\bpanel_smem\b|\d+|[()+*\s]", "", size)
        assert left == "", (size, left)
