"""Solve-phase kernels may be scheduled while the kernel before them in the
stream still runs (programmatic dependent launch).  Vectors that it writes must
not be read through the read-only path: __ldg, and loads through parameters that
are const __restrict__ (which the compiler turns into the same instruction),
promise data that does not change while the kernel is resident, and are ordered
after the wait by nothing but the compiler's habits.  Only what the setup wrote,
which ends with a synchronisation, may be read that way.  (Read from the
sources; no GPU needed.)
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2001_11533_gb300", "csrc")
FILES = ["blas.cu", "block.cu", "kuhn.cu", "mass.cu", "solver.cu", "sparse.cu", "state.cu", "transfer.cu", "fused.cu"]
# parameters that hold what the setup wrote: matrix values, indices, diagonals
SETUP = {"lo", "v", "cols", "inv", "invd", "invd32", "vinvd", "invd_c", "kappa", "sov", "vos", "sv", "fc"}
KERNEL = re.compile(r"__global__ void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(\w+)\(((?:[^()]|\([^()]*\))*)\)"
                    r"\s*\{(.*?)\n\}", re.S)


def dependent_kernels():
    for f in FILES:
        src = open(os.path.join(CSRC, f)).read()
        for name, params, body in KERNEL.findall(src):
            if re.search(r"pdl_enter|PDL_ENTER_LOADING|griddepcontrol\.wait", body):
                yield f, name, params


def test_the_sources_are_read():
    found = list(dependent_kernels())
    assert len(found) >= 55 and {f for f, _, _ in found} == set(FILES)


@pytest.mark.parametrize("f,name,params", list(dependent_kernels()), ids=lambda v: v if "*" not in v else "")
def test_no_read_only_vectors(f, name, params):
    ro = re.findall(r"const\s+[\w:<> ]+?\s*\*\s*__restrict__\s+(\w+)", params)
    assert not set(ro) - SETUP, (f, name, sorted(set(ro) - SETUP))


def test_no_ldg_in_solve_phase_sources():
    for f in FILES + ["spmv.cuh", "df.cuh", "clustercg.cuh", "util.cuh"]:
        src = re.sub(r"//.*", "", open(os.path.join(CSRC, f)).read())
        assert "__ldg(" not in src, f
