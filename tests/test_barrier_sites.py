"""All warps of a CTA meet a barrier at the same place in the source: CUDA promises
nothing for a __syncthreads() that some warps reach on another path.  (Read from
the sources; no GPU needed.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_11533_gb300", "csrc")


def body(src, name):
    m = re.search(r"\b" + name + r"\([^;{]*\)\s*\{(.*?)\n\}", src, re.S)
    return re.sub(r"//.*", "", m.group(1))


def test_rows_of_the_cluster_state_solve_wait_at_one_place():
    b = body(open(os.path.join(CSRC, "state.cu")).read(), "scg_row")
    assert b.count("scg_arrive(") == 1 and b.count("scg_wait(") == 1
    assert "return" not in b[:b.index("scg_wait(")].split("auto load")[0]
    assert "return" not in b[b.index("scg_arrive("):b.index("scg_wait(")]
