"""CG solves that run as one launch are timed and filed as such (kernel classes of
amgh_kernel_class_stats): one launch a solve, with the bytes of its iterations
and nothing else under their class; replayed levels file nothing there.
"""
import numpy as np
import pytest

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ONE = "cg_one_launch"


def stats(p, call):
    p.kernel_timing(True)
    call()
    out = p.kernel_class_stats()
    p.kernel_timing(False)
    return out


@pytest.mark.parametrize("precision", [0, 2])
def test_one_launch_solves_are_filed(precision):
    import torch
    from paper_2001_11533_gb300 import amgh
    p = amgh.Problem.from_workload(W.unit_square(33, jitter=0.2, cfg=77)).amg_setup(precision=precision, coarse_max=16)
    m, n = p.sizes["m"], p.sizes["n"]
    f, b = (torch.from_numpy(np.random.default_rng(k).standard_normal(k)).cuda() for k in (m, n))
    for call, vectors in ((lambda: p.state_solve_level(0, f, 1e-10), m), (lambda: p.mass_solve(0, b), n)):
        s = stats(p, call)
        # every iteration reads at least the matrix and the vectors of the level once
        assert s[ONE]["launches"] == 1 and s[ONE]["ms"] > 0 and s[ONE]["bytes"] > 10 * 8 * vectors
        assert all(v["launches"] == 0 for k, v in s.items() if k != ONE), s
    p.close()


def test_replayed_and_persistent_solves():
    import torch
    from paper_2001_11533_gb300 import amgh
    w = W.unit_square(129, jitter=0.2, cfg=77)
    for persistent in (0, 1):
        p = amgh.Problem.from_workload(w).amg_setup(precision=2, coarse_max=256, persistent_cg=persistent)
        b = torch.from_numpy(np.random.default_rng(1).standard_normal(p.sizes["n"])).cuda()
        s = stats(p, lambda: p.mass_solve(0, b))
        assert s[ONE]["launches"] == persistent and (s[ONE]["bytes"] > 0) == bool(persistent)
        assert (s["cg_spmv_l0"]["launches"] > 0) != bool(persistent)
        p.close()
