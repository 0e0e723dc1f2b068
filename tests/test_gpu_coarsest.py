"""Coarsest-grid inverse (nested dissection over the node rows) at its edges:
one block row, two, odd counts, rows of two DOFs, the widest rows of the block
path (80 DOFs) and the first that take the band factorisation, each through a
two-grid cycle against the oracle's.

The bar is that of the V-cycle parity tests: the GPU applies K_0^-1, the oracle
substitutes through the Cholesky factor, so they differ by up to about
kappa(K_0) eps.
"""

import numpy as np
import pytest
import torch

from oracle import fem, multigrid
from synth import BOTTOM, LEFT, RIGHT, TOP, dirichlet_design

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
EP = [1.0, 0.5, 0.25, 1e-9]


@pytest.mark.parametrize("nx0,ny0,fixed", [
    (1, 1, BOTTOM), (2, 1, BOTTOM | LEFT), (1, 2, BOTTOM), (3, 2, BOTTOM | TOP), (2, 3, LEFT), (1, 9, BOTTOM | LEFT),
    (5, 7, BOTTOM), (7, 16, BOTTOM | LEFT | RIGHT), (8, 33, BOTTOM), (16, 16, BOTTOM), (39, 3, BOTTOM),
    (40, 2, BOTTOM | LEFT), (40, 3, BOTTOM), (41, 6, BOTTOM | RIGHT)])
def test_two_grid_cycle(nx0, ny0, fixed):
    import paper_2301_07457_gb300 as mto

    nx, ny = 2 * nx0, 2 * ny0
    x = dirichlet_design(nx, ny, 4, seed=nx0 + ny0)
    E = fem.simp_moduli(x, EP, 3.0)
    lv = multigrid.build_hierarchy(nx, ny, E, fem.element_stiffness(0.3), fixed, 1)
    M = multigrid.vcycle_preconditioner(lv, 0.6, 2, 2)
    m = mto.Mesh(nx, ny, n_coarsen=1, fixed_edges=fixed)
    m.set_design(torch.from_numpy(x).to(DEV), EP, 3.0)
    m.set_design(torch.from_numpy(x).to(DEV), EP, 3.0)  # again over the first call's inverse
    r = np.random.default_rng(1).standard_normal((ny + 1, nx + 1, 2))
    r[fem.fixed_node_mask(nx, ny, fixed)] = 0.0
    z = m.apply_preconditioner(torch.from_numpy(r).to(DEV)).cpu().numpy()
    ref = np.zeros(r.size)
    ref[lv[-1].free] = M(r.ravel()[lv[-1].free])
    bar = max(1e-12, 20 * np.linalg.cond(lv[0].K.toarray()) * np.finfo(float).eps)
    assert np.linalg.norm(z.ravel() - ref) <= bar * np.linalg.norm(ref)
    m.close()
