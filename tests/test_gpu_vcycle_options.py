"""V-cycle and solves with other smoothing counts and damping (Alg. 1 with
theta_1 pre- and theta_2 post-smoothing sweeps of damped Jacobi), and the
W-cycle (gamma = 2, 3 below the finest grid), through the C ABI, against the
oracle.

The default (two and two, omega = 0.6) runs fused passes on the float32
levels and a fused first sweep on the finest level; other counts take the
separate-kernel paths (the first sweep from zero as a kernel of its own, the
prolongation sweep carrying the dot products, extra plain sweeps), and the
repeated coarse calls of a W-cycle start their smoothing from the last
iterate.  Bars as in
test_gpu_parity.py: float64 V-cycle max(1e-12, 20 kappa(K_0) eps), float32
V-cycle 2e-5 against the oracle's float64 V-cycle on the same bf16-rounded
moduli; solves reach the requested float64 true residual.
"""

import ctypes

import numpy as np
import pytest
import torch

from oracle import fem, multigrid, precision, solver
from synth import BOTTOM, dirichlet_design, load_top_edge

pytestmark = pytest.mark.gpu
EP = [1.0, 0.5, 0.25, 1e-9]
DEV = torch.device("cuda", 0)


@pytest.fixture(scope="module")
def mto():
    import paper_2301_07457_gb300 as m
    return m


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300)


def to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("nu1,nu2,omega", [(1, 1, 0.6), (1, 2, 0.6), (2, 1, 0.6), (3, 3, 0.6),
                                           (2, 2, 0.8), (3, 1, 0.5)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_vcycle_smoothing_counts(mto, prec, nu1, nu2, omega):
    nelx, nely, nc = 200, 136, 3
    x = dirichlet_design(nelx, nely, 4, seed=21)
    E = fem.simp_moduli(x, EP, 3.0)
    mesh = mto.Mesh(nelx, nely, n_coarsen=nc, precision=prec, nu1=nu1, nu2=nu2, omega=omega)
    mesh.set_design(to_dev(x), EP, 3.0)
    E_pre = precision.round_to_bf16(E) if prec == "mixed" else E
    lv = multigrid.build_hierarchy(nelx, nely, E_pre, fem.element_stiffness(0.3), BOTTOM, nc)
    M = multigrid.vcycle_preconditioner(lv, omega, nu1, nu2)
    r = np.random.default_rng(5).standard_normal((nely + 1, nelx + 1, 2))
    r[fem.fixed_node_mask(nelx, nely, BOTTOM)] = 0.0
    z = mesh.apply_preconditioner(to_dev(r)).cpu().numpy()
    ref = np.zeros(r.size)
    ref[lv[-1].free] = M(r.ravel()[lv[-1].free])
    kappa0 = np.linalg.cond(lv[0].K.toarray())
    bar64 = max(1e-12, 20 * kappa0 * np.finfo(float).eps)
    assert rel(z, ref) < (bar64 if prec == "fp64" else 2e-5), (rel(z, ref), kappa0)
    mesh.close()


@pytest.mark.parametrize("nu1,nu2", [(1, 1), (3, 3), (2, 1)])
def test_mixed_solve_smoothing_counts(mto, nu1, nu2):
    nelx = nely = 128
    x = dirichlet_design(nelx, nely, 4, seed=8)
    f = load_top_edge(nelx, nely)
    E = fem.simp_moduli(x, EP, 3.0)
    mesh = mto.Mesh(nelx, nely, n_coarsen=3, tol=1e-8, precision="mixed", nu1=nu1, nu2=nu2)
    mesh.set_design(to_dev(x), EP, 3.0)
    u, st = mesh.solve(to_dev(f))
    assert st["status"] == "MTO_OK", st
    assert solver.true_relative_residual(nelx, nely, E, f, u.cpu().numpy()) <= 1e-8
    mesh.close()


@pytest.mark.parametrize("gamma", [2, 3])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 2), (3, 1)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_w_cycle(mto, prec, nu1, nu2, gamma):
    # Five grids (192 x 128 down to 12 x 8): the coarse grids are called
    # 1, gamma and gamma^2 times per cycle.
    nelx, nely, nc = 192, 128, 4
    x = dirichlet_design(nelx, nely, 4, seed=22)
    E = fem.simp_moduli(x, EP, 3.0)
    mesh = mto.Mesh(nelx, nely, n_coarsen=nc, precision=prec, nu1=nu1, nu2=nu2, gamma=gamma)
    mesh.set_design(to_dev(x), EP, 3.0)
    E_pre = precision.round_to_bf16(E) if prec == "mixed" else E
    lv = multigrid.build_hierarchy(nelx, nely, E_pre, fem.element_stiffness(0.3), BOTTOM, nc)
    r = np.random.default_rng(6).standard_normal((nely + 1, nelx + 1, 2))
    r[fem.fixed_node_mask(nelx, nely, BOTTOM)] = 0.0
    z = mesh.apply_preconditioner(to_dev(r)).cpu().numpy()
    ref = np.zeros(r.size)
    ref[lv[-1].free] = multigrid.vcycle_preconditioner(lv, 0.6, nu1, nu2, gamma)(r.ravel()[lv[-1].free])
    vref = np.zeros(r.size)
    vref[lv[-1].free] = multigrid.vcycle_preconditioner(lv, 0.6, nu1, nu2)(r.ravel()[lv[-1].free])
    assert rel(ref, vref) > 1e-3  # the W-cycle is not the V-cycle here
    # Each coarsest solve (explicit inverse against Cholesky) contributes up
    # to ~kappa(K_0) eps, and the cycle carries each contribution to the
    # output without amplifying it: the V-cycle bar times the gamma^(nc-2)
    # coarsest solves of one W-cycle.
    kappa0 = np.linalg.cond(lv[0].K.toarray())
    bar64 = max(1e-12, 20 * kappa0 * np.finfo(float).eps * gamma ** (nc - 2))
    assert rel(z, ref) < (bar64 if prec == "fp64" else 2e-5), (rel(z, ref), kappa0)
    mesh.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_w_cycle_solve(mto, prec):
    nelx = nely = 128
    x = dirichlet_design(nelx, nely, 4, seed=9)
    f = load_top_edge(nelx, nely)
    E = fem.simp_moduli(x, EP, 3.0)
    mesh = mto.Mesh(nelx, nely, n_coarsen=4, tol=1e-8, precision=prec, gamma=2)
    mesh.set_design(to_dev(x), EP, 3.0)
    u, st = mesh.solve(to_dev(f))
    assert st["status"] == "MTO_OK", st
    assert solver.true_relative_residual(nelx, nely, E, f, u.cpu().numpy()) <= 1e-8
    if prec == "fp64":
        ref = solver.solve_pcgmg(nelx, nely, x, EP, 3.0, f, n_coarsen=4, tol=1e-8, gamma=2)
        assert abs(st["iters"] - ref["iters"]) <= 1, (st["iters"], ref["iters"])
    mesh.close()


@pytest.mark.parametrize("kind", ["galerkin", "rediscretize"])
@pytest.mark.parametrize("nx,ny,nc", [(32, 32, 3), (48, 40, 3), (136, 72, 3), (264, 136, 2), (96, 264, 3)])
def test_tiled_coarse_passes_equal_marching_ones(mto, nx, ny, nc, kind):
    """The small float32 levels run by tiles (a block per tile); a launch shape of one warp makes
    them march instead.  Both form every value by the same operations: equal bit for bit."""
    x = torch.from_numpy(dirichlet_design(nx, ny, 4, seed=nx)).cuda()
    r = torch.from_numpy(np.random.default_rng(ny).standard_normal((ny + 1, nx + 1, 2))).cuda()
    z = []
    for warps in (0, 1):
        m = mto.Mesh(nx, ny, n_coarsen=nc, precision="mixed", fixed_edges=mto.EDGE_BOTTOM | mto.EDGE_LEFT,
                     coarse_kind=kind)
        for l in range(1, nc):
            m.set_launch_shape(l, warps)
        m.set_design(x, [1.0, 0.5, 0.25, 1e-9], 3.0)
        z.append(m.apply_preconditioner(r))
        m.close()
    assert torch.equal(z[0], z[1])


@pytest.mark.parametrize("nu1,nu2", [(2, 2), (3, 3), (1, 2), (2, 1)])
@pytest.mark.parametrize("nx,ny,nc", [(8, 8, 1), (32, 24, 3), (62, 34, 1), (136, 72, 3)])
def test_mixed_cycle_between_the_callers_arrays(mto, nx, ny, nc, nu1, nu2):
    """With two sweeps or more, the first and last finest sweeps read and write the caller's
    float64 arrays.  The cycle is a float32 function of the rounded right-hand side on the free
    nodes, so rounding r first, non-finite values on clamped nodes, and an output that is the
    input (or overlaps it) change no bit."""
    x = torch.from_numpy(dirichlet_design(nx, ny, 4, seed=nx)).cuda()
    r = torch.from_numpy(np.random.default_rng(ny).standard_normal((ny + 1, nx + 1, 2))).cuda()
    m = mto.Mesh(nx, ny, n_coarsen=nc, precision="mixed", fixed_edges=mto.EDGE_BOTTOM | mto.EDGE_RIGHT,
                 nu1=nu1, nu2=nu2)
    m.set_design(x, EP, 3.0)
    z = m.apply_preconditioner(r)
    assert torch.equal(z, z.float().double()) and z.abs().max() > 0
    assert not z[0].any() and not z[:, -1].any()
    assert torch.equal(m.apply_preconditioner(r.float().double()), z)
    bad = r.clone()
    bad[0] = float("nan")
    bad[:, -1] = float("inf")
    assert torch.equal(m.apply_preconditioner(bad), z)
    for shift in (0, 2, 2 * (nx + 1) + 2):  # doubles from the input's start to the output's
        buf = torch.zeros(r.numel() + shift, dtype=torch.float64, device=DEV)
        buf[:r.numel()] = r.reshape(-1)
        st = m._lib.mto_apply_preconditioner(m._h, ctypes.c_void_p(buf.data_ptr()),
                                             ctypes.c_void_p(buf.data_ptr() + 8 * shift))
        assert st == 0
        torch.cuda.synchronize()
        assert torch.equal(buf[shift:], z.reshape(-1)), shift
    m.close()


@pytest.mark.parametrize("nu1,nu2", [(2, 2), (2, 3), (3, 2)])
@pytest.mark.parametrize("nx,ny,nc", [(8, 8, 1), (32, 24, 2), (62, 34, 1), (264, 136, 3)])
def test_tiled_finest_mixed_passes_equal_marching_ones(mto, nx, ny, nc, nu1, nu2):
    """The same for the bf16 finest level; its dot products and |r|^2 are summed by tiles, so a
    solve follows the bars of the mixed solves (iterations +- 2, u to 1e-6)."""
    x = torch.from_numpy(dirichlet_design(nx, ny, 4, seed=nx)).cuda()
    r = torch.from_numpy(np.random.default_rng(ny).standard_normal((ny + 1, nx + 1, 2))).cuda()
    f = torch.from_numpy(load_top_edge(nx, ny)).cuda()
    z, u, it = [], [], []
    for warps in (0, 1):
        m = mto.Mesh(nx, ny, n_coarsen=nc, precision="mixed", tol=1e-10, nu1=nu1, nu2=nu2, rr_every=5)
        m.set_launch_shape(nc, warps)
        m.set_design(x, EP, 3.0)
        z.append(m.apply_preconditioner(r))
        uu, st = m.solve(f)
        assert st["status"] == "MTO_OK" and st["rel_res_true"] <= 1e-10, st
        u.append(uu)
        it.append(st["iters"])
        m.close()
    assert torch.equal(z[0], z[1])
    assert abs(it[0] - it[1]) <= 2, it
    assert rel(u[0].cpu().numpy(), u[1].cpu().numpy()) < 1e-6
