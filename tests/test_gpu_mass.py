"""The one-launch mass CG (csrc/mass.cu) at the edges of its forms: one CTA, a
cluster, 8 or 16 entries a lane, 1 to 32 lanes a row, the last level that fits
and the first that does not.

Tolerance: the loop stops on its recursive residual, ||r|| <= tol ||b||; the true
residual differs from it by the rounding of ~40 updates (double-float: 40 x
2^-44 ~ 2e-12 of ||b||; FP64 far less), so with tol = 1e-11 the residual of the
answer, formed in FP64 from the level's own matrix, is at most 2e-11.
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


def problem(mesh, N, precision):
    from paper_2001_11533_gb300 import amgh
    w = W.unit_square(N, jitter=0.2, cfg=77) if mesh == "square" else W.cube_ball(N, contrast=0.5)
    p = amgh.Problem.from_workload(w).amg_setup(precision=precision, coarse_max=16)
    p.set_solve_opts(mass_tol=TOL)
    return p


# 128^2 = 16 CTAs of 1024 lanes, 129^2 is past it; 64^2 and 91^2 straddle the
# forms below; the cubes' coarse levels have rows of 25 to 100 entries
@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("mesh,N", [("square", 3), ("square", 16), ("square", 23), ("square", 64), ("square", 65),
                                    ("square", 91), ("square", 128), ("square", 129), ("cube", 6), ("cube", 17)])
def test_residual(mesh, N, precision):
    p = problem(mesh, N, precision)
    for level, n in enumerate(p.sizes["control"]):
        rp, ci, v, shape = p.matrix("Mu", level)
        M = sp.csr_matrix((v, ci, rp), shape=shape)
        b = np.random.default_rng(N + level).standard_normal(n)
        for scale in (1.0, 1e-120):   # a square of (r, z) would underflow at the second
            x, it = p.mass_solve(level, cuda(scale * b))
            x = x.cpu().numpy() / scale
            assert 0 < it <= 100
            assert np.linalg.norm(M @ x - b) <= 2 * TOL * np.linalg.norm(b), (level, n, scale)
        x, it = p.mass_solve(level, cuda(np.zeros(n)))
        assert it == 0 and not x.any()
    p.close()


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("N", [9, 33])
def test_statuses(N, precision):
    from paper_2001_11533_gb300 import amgh
    p = problem("square", N, precision)
    b = np.random.default_rng(N).standard_normal(p.sizes["n"])
    p.set_solve_opts(mass_tol=TOL, mass_max_iter=3)
    with pytest.raises(amgh.AmghError) as e:
        p.mass_solve(0, cuda(b))
    assert e.value.code == -5
    p.set_solve_opts(mass_tol=TOL)
    b[N] = np.nan
    with pytest.raises(amgh.AmghError) as e:
        p.mass_solve(0, cuda(b))
    assert e.value.code == -7
    p.close()
