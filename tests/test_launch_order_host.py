"""Kernels that may start before the kernel ahead of them in the stream has ended must not read what that one writes
through the read-only path, which keeps no order with the wait for it (a source check: an overlap cannot be forced)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_1263_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", ["stage_split.cuh", "stage_pair.cuh", "stage_march.cuh"])
def test_stage_kernels_that_start_early_use_ordinary_loads(name):
    s = source(name)
    assert "launch_early(" in s and "grid_wait()" in s
    assert "__ldg(" not in s and not re.search(r"\bld2<", s) and not re.search(r"\bGAcc<T, D>", s)


def test_words_that_kernels_hand_on_are_read_in_order():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "__ldcg(" not in source(os.path.basename(path)), path


def test_every_kernel_that_releases_the_next_waits_itself():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        s = source(os.path.basename(path))
        for body in re.split(r"__global__", s)[1:]:
            if "grid_launch_dependents();" in body:
                assert "grid_wait();" in body, path
