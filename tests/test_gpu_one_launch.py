"""Which form a state solve takes: one cluster launch (csrc/state.cu) on levels of
at most 2,048 rows whose hierarchy fits, exact zeros in the matrices or not
(regular 2D grids store a quarter of their entries as exact zeros, Kuhn cubes
about half), the replayed kernels elsewhere.  A cap of iterations above 10,000
takes the replayed form on every level, so both answer the same right side.

Tolerance: as in test_gpu_state.py, the residual formed in FP64 of a solve to
1e-10 is at most 2e-10 and the counts of both forms agree to one.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-10


def problem(mesh, N, precision, coarse_max):
    from paper_2001_11533_gb300 import amgh
    w = {"square": lambda: W.unit_square(N, cfg=77), "jittered": lambda: W.unit_square(N, jitter=0.2, cfg=77),
         "cube": lambda: W.cube_ball(N, contrast=0.5)}[mesh]()
    return amgh.Problem.from_workload(w).amg_setup(precision=precision, coarse_max=coarse_max)


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("mesh,N,coarse_max", [
    ("square", 14, 16), ("square", 33, 256), ("square", 47, 16), ("jittered", 33, 16), ("cube", 6, 16),
    ("cube", 9, 16), ("cube", 13, 256)])
def test_small_levels_are_one_launch(mesh, N, coarse_max, precision):
    import torch
    from paper_2001_11533_gb300 import amgh
    p = problem(mesh, N, precision, coarse_max)
    for level, n in enumerate(p.sizes["state"][:p.sizes["Ls"]]):
        rp, ci, v, shape = p.matrix("A", level)
        A = sp.csr_matrix((v, ci, rp), shape=shape)
        f = np.random.default_rng(N + level).standard_normal(n)
        ft = torch.from_numpy(f).cuda()
        counts, iters = [], []
        for cap in (10000, 10001):
            p.set_solve_opts(inner_max_iter=cap)
            n0 = amgh.launch_count()
            y, it = p.state_solve_level(level, ft, TOL)
            counts.append(amgh.launch_count() - n0)
            iters.append(it)
            assert np.linalg.norm(A @ y.cpu().numpy() - f) <= 2 * TOL * np.linalg.norm(f), (level, n, cap)
        assert counts[0] == 1 and counts[1] > 1, (level, n, counts)
        assert abs(iters[0] - iters[1]) <= 1, (level, n, iters)
    p.close()


@pytest.mark.parametrize("precision", [0, 2])
def test_first_level_past_the_cluster_is_replayed(precision):
    import torch
    from paper_2001_11533_gb300 import amgh
    p = problem("square", 49, precision, 256)
    n = p.sizes["state"][0]
    assert n == 2209
    n0 = amgh.launch_count()
    p.state_solve_level(0, torch.ones(n, dtype=torch.float64, device="cuda"), TOL)
    assert amgh.launch_count() - n0 > 1
    p.close()


@pytest.mark.parametrize("precision", [0, 2])
def test_falls_back_where_no_cluster_can_be_placed(precision):
    """A device that cannot place the clusters (here: none above one CTA counts)
    answers the same calls by the replayed kernels."""
    import torch
    from paper_2001_11533_gb300 import amgh
    p = problem("jittered", 33, precision, 16)
    p.set_solve_opts(mass_tol=TOL)
    rng = np.random.default_rng(33)
    for which, solve, n in (("A", lambda b: p.state_solve_level(0, b, TOL), p.sizes["m"]),
                            ("Mu", lambda b: p.mass_solve(0, b), p.sizes["n"])):
        rp, ci, v, shape = p.matrix(which, 0)
        A = sp.csr_matrix((v, ci, rp), shape=shape)
        f = rng.standard_normal(n)
        counts, iters = [], []
        try:
            for ctas in (-1, 1, -1):
                amgh.debug_cluster_ctas(ctas)
                n0 = amgh.launch_count()
                x, it = solve(torch.from_numpy(f).cuda())
                counts.append(amgh.launch_count() - n0)
                iters.append(it)
                assert np.linalg.norm(A @ x.cpu().numpy() - f) <= 2 * TOL * np.linalg.norm(f), (which, ctas)
        finally:
            amgh.debug_cluster_ctas(-1)
        assert counts[0] == counts[2] == 1 and counts[1] > 1, (which, counts)
        assert max(iters) - min(iters) <= 1, (which, iters)
    # block mass solves: one cluster a column, or the replayed block loop
    yd = torch.from_numpy(rng.standard_normal((3, p.sizes["n"]))).cuda()
    sopts = dict(tol=1e-8, inner_tol=TOL, mass_tol=TOL)
    u0, _, st0 = p.solve_block(yd, **sopts)
    try:
        amgh.debug_cluster_ctas(0)
        u1, _, st1 = p.solve_block(yd, **sopts)
    finally:
        amgh.debug_cluster_ctas(-1)
    assert st0 == 0 and st1 == 0
    # two outer CGs to a relative residual of 1e-8 on a Hessian whose M_u-scaled condition number is below 1 / beta = 100
    assert np.linalg.norm((u0 - u1).cpu().numpy()) <= 2e-6 * np.linalg.norm(u0.cpu().numpy())
    p.close()


def test_cluster_hook_rejects_bad_values():
    from paper_2001_11533_gb300 import amgh
    with pytest.raises(amgh.AmghError) as e:
        amgh.debug_cluster_ctas(-2)
    assert e.value.code == -1
