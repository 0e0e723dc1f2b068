"""The float64 sweeps in fixed point at their edges: strip and row remainders of
both kernels (a row per warp on small grids, marching tasks otherwise), values
far apart in size, moduli down to zero, non-finite input.

Bars: an operator row sums at most 18 products; float64 evaluation and the
fixed-point one both stay within a few eps of sum |K_ij| |v_j|, so 1e-14 of
that sum is allowed (about 45 eps).  Where rows span more than the scale of a
warp's window holds (about 2^60), that window's largest |K| |v| takes the
place of the row's own, at 2^-60.
"""

import numpy as np
import pytest
import torch

from oracle import fem, multigrid
from synth import BOTTOM, LEFT, RIGHT, dirichlet_design

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
EP = [1.0, 0.5, 0.25, 1e-9]
MARCH, ROWS = 1, 0  # target warps of a launch: one (long marching tasks), or a full wave (a row per warp here)


@pytest.fixture(scope="module")
def mto():
    import paper_2301_07457_gb300 as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def build(mto, nx, ny, fixed, x, prec="fp64", warps=ROWS):
    m = mto.Mesh(nx, ny, n_coarsen=1, fixed_edges=fixed, precision=prec)
    for l in (-1, 0, 1):
        m.set_launch_shape(l, warps)
    m.set_design(dev(x), EP, 3.0)
    return m


@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("nx,ny,fixed", [
    (2, 2, BOTTOM), (12, 4, BOTTOM), (14, 6, BOTTOM | LEFT), (16, 2, LEFT), (26, 8, BOTTOM), (28, 30, BOTTOM | RIGHT),
    (30, 50, BOTTOM), (58, 42, BOTTOM), (60, 10, RIGHT), (74, 34, BOTTOM | LEFT | RIGHT)])
def test_operator_and_cycle(mto, nx, ny, fixed, warps):
    x = dirichlet_design(nx, ny, 4, seed=nx + ny)
    lv = multigrid.build_hierarchy(nx, ny, fem.simp_moduli(x, EP, 3.0), fem.element_stiffness(0.3), fixed, 1)
    m = build(mto, nx, ny, fixed, x, warps=warps)
    rng = np.random.default_rng(nx * ny)
    for l in range(2):
        v = rng.standard_normal(m.level_shape(l))
        y = m.apply_operator(l, dev(v)).cpu().numpy().ravel()
        free, K = lv[l].free, lv[l].K
        ref = np.zeros(y.size)
        ref[free] = K @ v.ravel()[free]
        bar = np.zeros(y.size)
        bar[free] = abs(K) @ abs(v.ravel()[free])
        assert np.all(np.abs(y - ref) <= 1e-14 * bar)
    M = multigrid.vcycle_preconditioner(lv, 0.6, 2, 2)
    r = rng.standard_normal((ny + 1, nx + 1, 2))
    r[fem.fixed_node_mask(nx, ny, fixed)] = 0.0
    z = m.apply_preconditioner(dev(r)).cpu().numpy().ravel()
    ref = np.zeros(z.size)
    ref[lv[1].free] = M(r.ravel()[lv[1].free])
    tol = max(1e-12, 20 * np.linalg.cond(lv[0].K.toarray()) * np.finfo(float).eps)
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref)
    m.close()


@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("scale", ["tiny", "huge", "spread", "subnormal"])
def test_sizes_of_values(mto, warps, scale):
    nx, ny, fixed = 40, 22, BOTTOM
    x = dirichlet_design(nx, ny, 4, seed=4)
    x[:, 5:9, 3:30] = 0.0
    x[3, 5:9, 3:30] = 1.0  # a void block: moduli 1e-9 beside solids
    x[:, 15, 10] = 0.0     # an element without material
    E = fem.simp_moduli(x, EP, 3.0)
    K = fem.assemble(nx, ny, E, fem.element_stiffness(0.3)).toarray()
    free = fem.free_dofs(nx, ny, fixed)
    rng = np.random.default_rng(2)
    v = rng.standard_normal((ny + 1, nx + 1, 2))
    # Powers of two, so that scaling is exact in the reference too.
    if scale == "spread":
        v *= 2.0 ** rng.integers(-30, 31, v.shape)
    s = {"tiny": 2.0 ** -960, "huge": 2.0 ** 1000, "spread": 1.0, "subnormal": 2.0 ** -1060}[scale]
    m = build(mto, nx, ny, fixed, x, warps=warps)
    w = v * s  # rounded where subnormal
    y = m.apply_operator(1, dev(w)).cpu().numpy().ravel()
    vv = np.zeros(v.size)
    vv[free] = (w / s if scale == "subnormal" else v).ravel()[free]
    ref, bar = np.zeros(v.size), np.zeros(v.size)
    ref[free], bar[free] = (K @ vv)[free], (abs(K) @ abs(vv))[free]
    err = np.abs(y / s - ref)
    floor = 2.0 ** -60 * np.abs(vv).max() * abs(K).max() + (0.0 if scale != "subnormal" else 1.01 * 5e-324 / s)
    assert np.all(err <= 1e-14 * bar + floor)
    m.close()


@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_values_reach_their_neighbours_only(mto, warps, value):
    nx, ny, fixed = 64, 40, BOTTOM
    x = dirichlet_design(nx, ny, 4, seed=9)
    m = build(mto, nx, ny, fixed, x, warps=warps)
    v = np.random.default_rng(3).standard_normal((ny + 1, nx + 1, 2))
    good = m.apply_operator(1, dev(v)).cpu().numpy()
    for j, i, c in ((1, 0, 0), (20, 29, 1), (ny, nx, 0), (33, 14, 1)):
        w = v.copy()
        w[j, i, c] = value
        y = m.apply_operator(1, dev(w)).cpu().numpy()
        near = np.zeros((ny + 1, nx + 1), bool)
        near[max(j - 1, 0):j + 2, max(i - 1, 0):i + 2] = True
        near[0] = False  # clamped: zero whatever the neighbours
        assert not np.isfinite(y[near]).any()
        assert np.isfinite(y[~near]).all()
        assert np.allclose(y[~near], good[~near], rtol=1e-12, atol=1e-12)
    m.close()


@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("nc", [1, 3])
def test_cycle_is_linear_in_scale_and_passes_nan_on(mto, warps, nc):
    """Small levels run their two-stage passes by tiles (ROWS) or sweep by sweep in marching tasks.
    A power of two on the input comes out on the output up to the rounding of each scale's last
    bits; a non-finite residual reaches every free node through the coarsest solve."""
    nx, ny, fixed = 72, 40, BOTTOM
    m = mto.Mesh(nx, ny, n_coarsen=nc, fixed_edges=fixed)
    for l in range(-1, nc + 1):
        m.set_launch_shape(l, warps)
    m.set_design(dev(dirichlet_design(nx, ny, 4, seed=5)), EP, 3.0)
    r = np.random.default_rng(8).standard_normal((ny + 1, nx + 1, 2))
    r[0] = 0.0
    z = m.apply_preconditioner(dev(r)).cpu().numpy()
    for s in (2.0 ** -900, 2.0 ** 900):
        zs = m.apply_preconditioner(dev(r * s)).cpu().numpy() / s
        assert np.linalg.norm(zs - z) <= 1e-12 * np.linalg.norm(z)
    for value in (np.nan, np.inf):
        bad = r.copy()
        bad[17, 33, 1] = value
        zb = m.apply_preconditioner(dev(bad)).cpu().numpy()
        assert not np.isfinite(zb[1:]).any() and np.all(zb[0] == 0.0)
    m.close()
