"""Orderings of the kernels that no result need show, read from the sources.  A
warp vote (__any_sync) orders no memory, so the places that vote between reads
of shared memory and the writes that replace what was read must have a barrier
too."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2512_08611_gb300", "csrc")
# votes on values in registers, with registers, shuffles or atomics behind them
REGISTERS_ONLY = ("theta_one_element(", "b != 0")


def votes():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        lines = [re.sub(r"//.*", "", x).strip() for x in open(path)]
        lines = [x for x in lines if x]
        for k, line in enumerate(lines):
            if re.search(r"__(any|all|ballot)_sync\(", line):
                yield os.path.basename(path), lines[k - 1], line


def test_votes_that_guard_shared_memory_have_a_barrier():
    found = list(votes())
    assert found
    for name, before, line in found:
        if any(r in line for r in REGISTERS_ONLY):
            continue
        assert before.endswith("__syncwarp();") and "?" not in line, (name, line)


def test_stage_votes_are_barriers():
    # the three kernels with one exchange area for all stages of an element
    for name in ("local_2d.cuh", "step_1d.cuh", "kernels_adj2d.cu"):
        text = open(os.path.join(CSRC, name)).read()
        assert "warp_barrier_or(" in text, name


def test_loops_over_tiles_release_the_next_kernel_last():
    # launch.h: the next kernel of the stream is let in when the blocks are
    # about to leave, not in the first of many steps or tiles
    text = open(os.path.join(CSRC, "step_1d.cuh")).read()
    assert re.findall(r"\n( *.*chain_end\(\);)", text) == ["  if (last) chain_end();"]
    assert "k + 1 == L.steps)" in text and "wi + gridDim.x >= B.nwork)" in text
