"""Settings that belong to a device are made for the device in use: kernel attributes
(shared memory above 48 KB, the L1 carve-out) hold for the current device only, so no
source guards them by a flag kept for the whole process, and their result is looked at."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1810_09898_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


@pytest.mark.parametrize("name", SOURCES)
def test_no_kernel_attribute_behind_a_process_wide_flag(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert not re.search(r"\bstatic\s+(std::atomic<)?bool\b", text)
    for m in re.finditer(r"cudaFuncSetAttribute\(", text):
        assert text[:m.start()].rstrip().endswith("check_cuda("), text[m.start():m.start() + 120]
