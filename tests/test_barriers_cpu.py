"""Barriers of the bispectrum task body, read from its source: the stage barrier is reached by a CTA's warps from
different instantiations of the frame loop, so it has to be one that counts arrivals by number, not __syncthreads()."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_stage_barrier_is_numbered():
    src = open(os.path.join(ROOT, "paper_1701_00581_gb300", "csrc", "sm_bispec_tile.cuh")).read()
    src = re.sub(r"//[^\n]*", "", src)
    start = src.index("auto next_stage")
    loops = src[start:src.index("for (int pass = 0", start)]      # next_stage and the loops made per column count
    assert "__syncthreads" not in loops
    assert re.search(r'"bar\.sync 1, %0;" :: "n"\(THREADS\) : "memory"', loops)
    # every branch of a pass goes through all of its stages
    branches = src[src.index("for (int pass = 0", start):]
    assert branches.count("for (int st = 0; st < nst; ++st) next_stage(st);") == 1
    assert loops.count("for (int st = 0; st < nst; ++st)") == 1 and loops.count("next_stage(st)") == 1
    assert not re.search(r"\b(break|return|continue)\b", loops[loops.index("for (int st = 0;"):loops.index("if (quad < 0)")])
