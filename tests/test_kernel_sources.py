"""Rules that a compiler may break without a word, checked on the kernels' text."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_13587_b200", "csrc")
# Waits that every lane of a warp leaves by itself; instructions that a whole warp has to execute together; what brings its lanes together
# before them (shuffles, votes and elections name their lanes).
WAIT = r"(?<!bool )\b(?:wait_or_abort|mbar_try_wait_cluster|mbar_wait)\("
ALIGNED = r"\b(?:cluster_wait|cluster_arrive|cluster_arrive_relaxed|cluster_sync|tmem_ld\d+|tmem_dealloc|ldsm4t?|mma16816)\("
MEET = r"\b(?:__syncwarp|__syncthreads|__syncthreads_or|named_bar_all|named_bar_sync|__shfl_xor_sync|elect_one|mma_bf16_k64|mma_pair_k64)\("


def _code(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu"))))
def test_lanes_meet_behind_a_wait(name):
    code = _code(os.path.join(CSRC, name))
    for wait in re.finditer(WAIT, code):
        line = code[code.rfind("\n", 0, wait.start()) + 1:wait.start()]
        if re.search(r"__all_sync\(|named_bar_all\(", line):
            continue
        behind = re.search(ALIGNED, code[wait.end():])
        if behind:
            between = code[wait.end():wait.end() + behind.start()]
            assert re.search(MEET, between), (name, code.count("\n", 0, wait.start()) + 1, behind.group())


def test_no_mask_of_lanes_that_happen_to_be_there():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "__activemask" not in _code(path), path
