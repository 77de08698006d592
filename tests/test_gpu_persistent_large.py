"""The single-column persistent mass CG (persistent_cg = 1, precision 2) on a level
that is too large for the one-cluster form of csrc/mass.cu: 129^2 = 16,641 rows
of seven entries, past 16 CTAs of 1,024 lanes.  (test_gpu_persistent.py's levels
all fit a cluster, which comes first.)  Four launches a solve: norm, start, all
iterations, output.

Tolerance: as in test_gpu_mass.py, the true residual of a solve to 1e-11 is at
most 2e-11; the mass matrix with its Jacobi scaling has a condition number below
100 on these meshes, so two such solutions differ by less than 1e-9.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11


def cuda(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


def problem(N, **opts):
    from paper_2001_11533_gb300 import amgh
    w = W.unit_square(N, jitter=0.2, cfg=77)
    p = amgh.Problem.from_workload(w).amg_setup(precision=2, coarse_max=256, **opts)
    p.set_solve_opts(mass_tol=TOL)
    return p


@pytest.mark.parametrize("N", [129, 257])
def test_persistent_matches_replay_and_residual(N):
    from paper_2001_11533_gb300 import amgh
    per, ref = problem(N, persistent_cg=1), problem(N)
    n = per.sizes["n"]
    rp, ci, v, shape = per.matrix("Mu", 0)
    M = sp.csr_matrix((v, ci, rp), shape=shape)
    b = np.random.default_rng(N).standard_normal(n)
    n0 = amgh.launch_count()
    x, it = per.mass_solve(0, cuda(b))
    n1 = amgh.launch_count()
    y, it0 = ref.mass_solve(0, cuda(b))
    assert n1 - n0 == 4 and amgh.launch_count() - n1 > 4   # persistent; replayed
    x, y = x.cpu().numpy(), y.cpu().numpy()
    assert 0 < it and abs(it - it0) <= 2
    assert np.linalg.norm(M @ x - b) <= 2 * TOL * np.linalg.norm(b)
    assert np.linalg.norm(x - y) <= 1e-9 * np.linalg.norm(y)
    per.close()
    ref.close()


def test_statuses_as_on_small_levels():
    """An iteration cap that is reached, a NaN and a barrier that gives up are
    reported by this form too, and the next solve is the clean one again."""
    from paper_2001_11533_gb300 import amgh
    p = problem(129, persistent_cg=1)
    b = np.random.default_rng(1).standard_normal(p.sizes["n"])
    clean = p.mass_solve(0, cuda(b))[0].cpu().numpy()

    def code(rhs):
        with pytest.raises(amgh.AmghError) as e:
            p.mass_solve(0, cuda(rhs))
        return e.value.code

    p.set_solve_opts(mass_tol=TOL, mass_max_iter=3)
    assert code(b) == -5
    p.set_solve_opts(mass_tol=TOL)
    bad = b.copy()
    bad[7] = np.nan
    assert code(bad) == -7
    try:
        amgh.debug_grid_polls(0)
        assert code(b) == amgh.ERR_TIMEOUT
    finally:
        amgh.debug_grid_polls(-1)
    assert np.array_equal(p.mass_solve(0, cuda(b))[0].cpu().numpy(), clean)
    p.close()


def test_batch_keeps_cooperative_launches_off_on_large_levels():
    """persistent_cg passed to a batch setup changes nothing, launch counts
    included, on a mesh whose finest mass solves do not fit a cluster."""
    from paper_2001_11533_gb300 import amgh
    ws = W.batch_squares(sizes=(129,), per_size=1, rhs=2)
    sopts = dict(tol=1e-8, inner_tol=1e-10, mass_tol=1e-8, precond_tol=1e-8, level_fallback=1)
    out = []
    for extra in ({}, dict(persistent_cg=1)):
        probs = [amgh.Problem.from_workload(w) for w in ws]
        batch = amgh.Batch(probs).setup(coarse_max=1000, precision=2, coarse_solve=2, **extra)
        n0 = amgh.launch_count()
        u, _, st = batch.solve([cuda(w.y_d) for w in ws], **sopts)
        assert st == 0
        out.append(([x.cpu().numpy() for x in u], amgh.launch_count() - n0))
    assert all(np.array_equal(a, b) for a, b in zip(out[0][0], out[1][0]))
    assert out[0][1] == out[1][1]


def test_second_setup_makes_new_work_space():
    """The work space of the persistent solves goes with the hierarchy that it
    was allocated beside: a second setup on the handle starts without it."""
    p, fresh = problem(129, persistent_cg=1), problem(129, persistent_cg=1)
    b = cuda(np.random.default_rng(2).standard_normal(p.sizes["n"]))
    p.mass_solve(0, b)
    p.amg_setup(precision=2, coarse_max=64, persistent_cg=1)
    p.amg_setup(precision=2, coarse_max=256, persistent_cg=1)
    x, it = p.mass_solve(0, b)
    y, it0 = fresh.mass_solve(0, b)
    assert it == it0 and np.array_equal(x.cpu().numpy(), y.cpu().numpy())
    p.close()
    fresh.close()
