"""A call on non-finite data leaves nothing behind for the next solve on the same mesh."""

import numpy as np
import pytest
import torch

from oracle import fem, solver
from synth import dirichlet_design, load_top_edge

pytestmark = pytest.mark.gpu
EP = [1.0, 0.5, 0.25, 1e-9]
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,nc,warps", [(64, 2, 0), (64, 2, 1), (512, 5, 0)])  # tiles, marching tasks, both
@pytest.mark.parametrize("call", ["operator", "operator in place", "preconditioner", "solve"])
def test_solve_after_non_finite_input(call, n, nc, warps, prec):
    import paper_2301_07457_gb300 as mto
    from paper_2301_07457_gb300 import _lib
    x, f = dirichlet_design(n, n, 4, seed=n), load_top_edge(n, n)
    m = mto.Mesh(n, n, n_coarsen=nc, precision=prec, tol=1e-8)
    for l in range(-1, nc + 1):
        m.set_launch_shape(l, warps)
    m.set_design(torch.from_numpy(x).to(DEV), EP, 3.0)
    v = torch.full((n + 1, n + 1, 2), float("nan"), dtype=torch.float64, device=DEV)
    if call == "operator":
        m.apply_operator(nc, v)
    elif call == "operator in place":  # goes through the context's own vectors
        lib = _lib.load()
        assert lib.mto_apply_operator(m._h, nc, 0, v.data_ptr(), v.data_ptr()) == 0
    elif call == "preconditioner":
        m.apply_preconditioner(v)
    else:
        m.solve(v, raise_on_failure=False)
    u, st = m.solve(torch.from_numpy(f).to(DEV))
    E = fem.simp_moduli(x, EP, 3.0)
    assert st["converged"] and solver.true_relative_residual(n, n, E, f, u.cpu().numpy()) <= 2e-8
    m.close()
