"""Warps that wait at different places of the source do so by PTX barriers, which
count the warps that arrive wherever they do; CUDA defines __syncthreads() only
where all of them reach the same one.  (Read from the sources; no GPU needed.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_11533_gb300", "csrc")


def body(src, name):
    m = re.search(r"\b" + name + r"\([^;{]*\)\s*\{(.*?)\n\}", src, re.S)
    return re.sub(r"//.*", "", m.group(1))


def test_waits_of_the_cluster_state_solve_are_ptx_barriers():
    src = open(os.path.join(CSRC, "state.cu")).read()
    row, wait = body(src, "scg_row"), body(src, "scg_wait")
    assert row.count("scg_arrive(") == 1 and row.count("scg_wait(") == 2  # with and without entries
    assert "__syncthreads" not in row and "__syncthreads" not in wait
    assert "barrier.cta.sync.aligned 0;" in wait and "barrier.cluster.wait" in wait
