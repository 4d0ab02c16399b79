"""The paths that the tensor-core kernels take when a wait gives up, read from their
sources: making a wait expire there would be a GPU left hanging if the path were
wrong, so the rules that keep it right are checked on the text.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2602_08642_gb300", "csrc")
KERNELS = ("conv_tc.cu", "wgrad_tc.cu")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", KERNELS)
def test_waits_before_warp_wide_code_have_one_answer_per_warp(name):
    """Only the threads that fill stages wait by themselves (for a stage or a coarse
    buffer to be free, or for a coarse box) and may leave one by one; accumulators
    and full stages are waited for by warps that go on with warp-wide loads, votes
    and __syncwarp, so their lanes have to leave together."""
    waits = re.findall(r"tc::(mbar_wait\w*)\(\s*&?([\w.]+)[^;]*?,\s*(abort_flag|nullptr)\)",
                       _source(name))
    alone = {bar for fn, bar, flag in waits if fn == "mbar_wait" and flag == "abort_flag"}
    assert alone and alone <= {"bars.empty", "bars.updone", "bars.upfull"}
    together = [bar for fn, bar, _ in waits if fn == "mbar_wait_warp"]
    assert "bars.accf" in together and len(together) >= 3


@pytest.mark.parametrize("name", KERNELS)
def test_copies_and_mmas_are_waited_for_on_every_path(name):
    """A role that never gave up itself may still have copies or MMAs in flight when
    another one did; so the waits before it leaves hang on what it issued (`pending`,
    `acc`, the counts in the loops), not on its own success."""
    src = _source(name)
    assert set(re.findall(r"if \(!ok\b[^{;]*[{;]", src)) <= {"if (!ok) break;"}
    assert not re.search(r"if \(issued\b[^)]*<", src)
    assert not re.search(r"\belse if \(acc\)", src)
    drains = re.findall(r"if \((\w+)\) \{\s*tc::mma_commit\(&bars\.drain", src)
    assert len(drains) == src.count("mma_commit(&bars.drain") and set(drains) <= {"pending", "acc"}
