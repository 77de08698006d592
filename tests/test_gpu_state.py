"""The one-launch state CG (csrc/state.cu) at the edges of its forms: one CTA, a
cluster, the last level that fits and the first that does not, a level that is
the dense coarsest one, smoothers of 1 to 3 steps, rows of one lane and of many.

Tolerance: the loop stops on its recursive residual, ||r|| <= tol ||b||; the true
residual differs from it by the rounding of at most ~40 updates (double-float:
40 x 2^-44 ~ 2e-12 of ||b||, times the ~10 by which ||A|| ||x|| exceeds ||b|| on
these levels; FP64 far less), so with tol = 1e-10 the residual of the answer,
formed in FP64 from the level's own matrix, is at most 2e-10.  V-cycles of other
row groupings round differently, so iteration counts agree to one with plain CG
preconditioned by the level's own V-cycle, here in numpy.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-10


def cuda(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


def problem(mesh, N, precision, **opts):
    from paper_2001_11533_gb300 import amgh
    w = W.unit_square(N, jitter=0.2, cfg=77) if mesh == "square" else W.cube_ball(N, contrast=0.5)
    return amgh.Problem.from_workload(w).amg_setup(precision=precision, **{"coarse_max": 16, **opts})


# 47^2 = 2,209 state rows are past the last level that fits, 45^2 = 2,025 are the
# last of the squares that do; 3^2 to 13^2 run as one CTA (FP32)
@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("mesh,N,opts", [
    ("square", 5, {}), ("square", 13, {}), ("square", 14, {}), ("square", 23, dict(coarse_max=1000)),
    ("square", 33, {}), ("square", 33, dict(smooth_degree=1)), ("square", 33, dict(smooth_degree=3, smoother=1)),
    ("square", 47, {}), ("square", 49, {}), ("square", 65, dict(coarse_max=256)), ("cube", 9, {}), ("cube", 17, {})])
def test_residual_and_iterations(mesh, N, opts, precision):
    p = problem(mesh, N, precision, **opts)
    for level, n in enumerate(p.sizes["state"][:p.sizes["Ls"]]):
        rp, ci, v, shape = p.matrix("A", level)
        A = sp.csr_matrix((v, ci, rp), shape=shape)
        b = np.random.default_rng(N + level).standard_normal(n)
        for scale in (1.0, 1e-120):
            x, it = p.state_solve_level(level, cuda(scale * b), TOL)
            x = x.cpu().numpy() / scale
            assert np.linalg.norm(A @ x - b) <= 2 * TOL * np.linalg.norm(b), (level, n, scale)
            # the same loop, one launch at a time: V-cycle and product from the library
            y, r = np.zeros(n), b.copy()
            z = p.vcycle(level, cuda(r)).cpu().numpy()
            d, rz, k = z.copy(), r @ z, 0
            while np.linalg.norm(r) > TOL * np.linalg.norm(b):
                q = A @ d
                alpha = rz / (d @ q)
                y += alpha * d
                r -= alpha * q
                z = p.vcycle(level, cuda(r)).cpu().numpy()
                d, rz, k = z + (r @ z) / rz * d, r @ z, k + 1
            assert abs(it - k) <= 1, (level, n, it, k)
        x, it = p.state_solve_level(level, cuda(np.zeros(n)), TOL)
        assert it == 0 and not x.any()
    p.close()


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("N", [9, 33])
def test_statuses(N, precision):
    from paper_2001_11533_gb300 import amgh
    p = problem("square", N, precision)
    b = np.random.default_rng(N).standard_normal(p.sizes["m"])
    p.set_solve_opts(inner_max_iter=2)
    with pytest.raises(amgh.AmghError) as e:
        p.state_solve_level(0, cuda(b), TOL)
    assert e.value.code == -5
    p.set_solve_opts()
    b[N] = np.nan
    with pytest.raises(amgh.AmghError) as e:
        p.state_solve_level(0, cuda(b), TOL)
    assert e.value.code == -7
    p.close()


# a cap above which the loop is replayed (csrc/clustercg.cuh) instead: same answer
@pytest.mark.parametrize("cap", [10000, 10001])
@pytest.mark.parametrize("precision", [0, 2])
def test_iteration_caps(precision, cap):
    p = problem("square", 33, precision)
    p.set_solve_opts(inner_max_iter=cap, mass_max_iter=cap, mass_tol=TOL)
    for which, solve, n in (("A", lambda b: p.state_solve_level(0, b, TOL), p.sizes["m"]),
                            ("Mu", lambda b: p.mass_solve(0, b), p.sizes["n"])):
        rp, ci, v, shape = p.matrix(which, 0)
        A = sp.csr_matrix((v, ci, rp), shape=shape)
        b = np.random.default_rng(5).standard_normal(n)
        x, it = solve(cuda(b))
        assert 0 < it <= 100
        assert np.linalg.norm(A @ x.cpu().numpy() - b) <= 2 * TOL * np.linalg.norm(b)
    p.close()
