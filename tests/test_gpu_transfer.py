"""The transfers fused with the products beside them (csrc/transfer.cu), in every
arrangement of levels and smoother steps an FP32 V-cycle can have: coarsest
level directly below, one to three smoother steps, l1-Jacobi, unsmoothed
prolongators, 2D and 3D rows, and the largest level that is fused (257^2, 65,025
states) beside the smallest that is not (259^2).

The solve stops on its recursive residual, ||r|| <= tol ||f||.  The true residual
differs from it by the rounding of the updates and of y itself, at most about
40 x 2^-44 |A| |y| in double-float; |A| |y| / ||f|| grows with the squared mesh
width to about 1e4 here, so with tol = 1e-8 it is below 2e-8.  The V-cycle is the
FP64 one up to FP32 rounding, so the iteration counts differ by at most two.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-8

OPTS = [dict(), dict(max_levels=2), dict(smooth_degree=1), dict(smooth_degree=3), dict(smoother=0),
        dict(smooth_prolongator=0)]
CASES = [("square", 5, {}), ("square", 257, {}), ("square", 259, {}), ("cube", 17, {})]
CASES += [("lshape", 33, o) for o in OPTS] + [("cube", 9, o) for o in OPTS]


@pytest.mark.parametrize("mesh,N,opts", CASES)
def test_fp32_cycles_solve_every_level(mesh, N, opts):
    import torch
    from paper_2001_11533_gb300 import amgh
    w = {"square": lambda: W.unit_square(N, jitter=0.2, cfg=5), "lshape": lambda: W.lshape_checkerboard(N=N),
         "cube": lambda: W.cube_ball(N, contrast=0.5)}[mesh]()
    kw = dict(dict(coarse_max=16), **opts)
    p64 = amgh.Problem.from_workload(w).amg_setup(precision=0, **kw)
    p32 = amgh.Problem.from_workload(w).amg_setup(precision=2, **kw)
    for level, n in enumerate(p32.sizes["state"]):
        rp, ci, v, shape = p32.matrix("A", level)
        A = sp.csr_matrix((v, ci, rp), shape=shape)
        f = np.random.default_rng(level).standard_normal(n)
        ft = torch.from_numpy(f).cuda()
        y, it = p32.state_solve_level(level, ft, TOL)
        _, it64 = p64.state_solve_level(level, ft, TOL)
        assert np.linalg.norm(A @ y.cpu().numpy() - f) <= 2 * TOL * np.linalg.norm(f), (level, n)
        assert abs(it - it64) <= 2, (level, n, it, it64)
    p32.close()
    p64.close()
