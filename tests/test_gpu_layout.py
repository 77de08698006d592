"""Solve-phase CSR layouts (csrc/sparse.cu): exact zeros left out, column offsets
in int16 where every one fits.  A 33^3 cube has 35,937 control rows: in grid
order the offsets of its mass and coarse stiffness matrices fit, under a random
numbering those of the finest level do not.

The solves stop on their recursive residual; the true one, formed in FP64 from
the level's canonical matrix, differs by the rounding of the updates (below 1e-9
of ||f|| here, see test_gpu_transfer.py), so at tol = 1e-8 it is at most 2e-8.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2001_11533_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-8


def permuted(w, seed):
    """The same problem with its vertices renumbered at random."""
    n = w.n_vertices
    new = np.random.default_rng(seed).permutation(n)
    coords, dirichlet, yd = np.empty_like(w.coords), np.empty_like(w.dirichlet), np.empty_like(w.y_d)
    coords[new], dirichlet[new], yd[new] = w.coords, w.dirichlet, w.y_d
    return W.Workload(w.name, w.dim, coords, new[w.elements].astype(np.int32), dirichlet, w.kappa, w.beta, yd)


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("order", ["grid", "random"])
@pytest.mark.parametrize("N", [6, 33])
def test_products_in_every_layout(N, order, precision):
    import torch
    from paper_2001_11533_gb300 import amgh
    w = W.cube_ball(N, contrast=0.5)
    if order == "random":
        w = permuted(w, N)
    p = amgh.Problem.from_workload(w).amg_setup(precision=precision, coarse_max=16)
    p.set_solve_opts(mass_tol=TOL)
    rng = np.random.default_rng(N)
    for which, hier in (("A", "state"), ("Mu", "control")):
        for level, n in enumerate(p.sizes[hier]):
            rp, ci, v, shape = p.matrix(which, level)
            A = sp.csr_matrix((v, ci, rp), shape=shape)
            f = rng.standard_normal(n)
            ft = torch.from_numpy(f).cuda()
            y = (p.state_solve_level(level, ft, TOL) if which == "A" else p.mass_solve(level, ft))[0]
            assert np.linalg.norm(A @ y.cpu().numpy() - f) <= 2 * TOL * np.linalg.norm(f), (which, level, n)
    p.close()
