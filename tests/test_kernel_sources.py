"""What can only be read off the kernels' sources: a wait that gives up needs half a second of a copy that never ends, which no test may
bring about."""
import os
import re

import pytest

from paper_2601_13143_b200 import build

# Kernels whose warps vote or shuffle after a bounded wait.  mbar_wait_bounded answers every lane for itself: lanes that leave on its
# answer are missing in the next full-mask operation.
WHOLE_WARP = ["compact.cu", "score_narrow.cu"]


@pytest.mark.parametrize("name", WHOLE_WARP)
def test_a_warp_that_votes_decides_on_one_answer(name):
    with open(os.path.join(build.CSRC, name)) as f:
        source = re.sub(r"//[^\n]*", "", f.read())
    assert "_sync(0xFFFFFFFFu" in source and "mbar_wait_warp(" in source
    for decision in re.findall(r"(?:if \(!?|= |while \(!?|&& !?)ptx::mbar_wait_bounded\(", source):
        pytest.fail(f"{name} decides on the answer of a single lane: {decision}")


def _kernels(name):
    with open(os.path.join(build.CSRC, name)) as f:
        source = re.sub(r"//[^\n]*", "", f.read())
    return re.split(r"\b__global__\b", source)[1:]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(build.CSRC) if f.endswith(".cu")))
def test_a_block_that_gives_up_waits_for_its_copies(name):
    """Copies that a kernel has asked for write into its block's shared memory, which is the next block's as soon as it exits: where a
    wait for them gives up, they are waited for once more, with a flag of its own that no other warp's giving up sets."""
    for kernel in _kernels(name):
        if re.search(r"\b(?:bulk_load|tma_load_\w+)\(", kernel):
            assert re.search(r"mbar_wait_bounded\([^;]*&never\)", kernel) or "drain_loads(" in kernel, f"{name}: {kernel[:120]}"


@pytest.mark.parametrize("name", ["score_rows.cu", "prune_few.cu"])
def test_warps_that_shuffle_behind_a_bounded_wait_decide_on_one_answer(name):
    test_a_warp_that_votes_decides_on_one_answer(name)
