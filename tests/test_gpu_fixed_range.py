"""Float64 operator and V-cycle where moduli or values of one neighbourhood are
further apart than a shared fixed-point scale holds.

Bars: a row of K v within 1e-14 of its own sum |K_ij| |v_j|, as in float64 (at
most 18 products; about 45 eps), whatever lies beside it.  V-cycle: the
oracle's own cycle is within 3e-15 (norm) of one in extended precision at every
ratio below, so 1e-13 of the norm is allowed, and 1e-12 on the stiff nodes alone.
"""

import numpy as np
import pytest
import torch

from oracle import fem, multigrid, solver
from synth import BOTTOM, LEFT, dirichlet_design, load_top_edge

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
MARCH, ROWS = 1, 0  # one long marching task, or a full wave (a row per warp and tiles here)
RATIOS = [1e-9, 1e-12, 1e-15, 1e-18, 1e-21, 1e-24, 1e-27, 1e-30]


@pytest.fixture(scope="module")
def mto():
    import paper_2301_07457_gb300 as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def soft_design(nx, ny, kind):
    """Two phases; the second (soft) one fills a block or the upper left quadrant."""
    x = np.zeros((2, ny, nx))
    if kind == "block":
        x[1, ny // 4:3 * ny // 4, nx // 4:3 * nx // 4] = 1.0
    else:
        x[1, ny // 2:, :nx // 2] = 1.0
    x[0] = 1.0 - x[1]
    return x


def build(mto, nx, ny, nc, x, Es, fixed=BOTTOM, warps=ROWS, **kw):
    m = mto.Mesh(nx, ny, n_coarsen=nc, fixed_edges=fixed, **kw)
    for l in range(-1, nc + 1):
        m.set_launch_shape(l, warps)
    m.set_design(dev(x), Es, 3.0)
    return m


def check_rows(m, lv, l, v, scale=1.0):
    y = m.apply_operator(l, dev(v * scale)).cpu().numpy().ravel() / scale
    free, K = lv[l].free, lv[l].K
    ref, bar = np.zeros(y.size), np.zeros(y.size)
    ref[free], bar[free] = K @ v.ravel()[free], abs(K) @ abs(v.ravel()[free])
    assert np.all(np.abs(y - ref) <= 1e-14 * bar)


@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("kind", ["block", "quadrant"])
@pytest.mark.parametrize("ratio", RATIOS)
def test_soft_beside_stiff(mto, ratio, kind, warps):
    nx, ny, fixed = 44, 24, BOTTOM | LEFT
    x, Es = soft_design(nx, ny, kind), [1.0, ratio]
    lv = multigrid.build_hierarchy(nx, ny, fem.simp_moduli(x, Es, 3.0), fem.element_stiffness(0.3), fixed, 2)
    m = build(mto, nx, ny, 2, x, Es, fixed, warps)
    rng = np.random.default_rng(nx)
    for l in range(3):
        v = rng.standard_normal(m.level_shape(l))
        check_rows(m, lv, l, v)
        # Both components of a node alike: a coupling that vanishes in exact arithmetic (u_x to u_y along
        # an edge) leaves rounding of the larger one in float64 too, outside such a bar.
        v = rng.choice([-1.0, 1.0], v.shape) * rng.uniform(0.5, 1.0, v.shape)
        v *= 2.0 ** rng.integers(-40, 41, v.shape[:2] + (1,))
        check_rows(m, lv, l, v)
    r = rng.standard_normal((ny + 1, nx + 1, 2))
    r[fem.fixed_node_mask(nx, ny, fixed)] = 0.0
    z = m.apply_preconditioner(dev(r)).cpu().numpy().ravel()[lv[2].free]
    ref = multigrid.vcycle_preconditioner(lv, 0.6, 2, 2)(r.ravel()[lv[2].free])
    assert np.linalg.norm(z - ref) <= 1e-13 * np.linalg.norm(ref)
    stiff = lv[2].diag > 0.1
    assert np.linalg.norm((z - ref)[stiff]) <= 1e-12 * np.linalg.norm(ref[stiff])
    m.close()


@pytest.mark.parametrize("k", [33, 34, 35, 36, 37])
@pytest.mark.parametrize("warps", [MARCH, ROWS])
def test_coarse_rows_near_the_line(mto, warps, k):
    """Coarse rows of a block 2^-k as stiff as its surroundings, against extended precision: root mean
    square error over a row's own terms.  Float64 sweeps show 9.2e-17 here at every ratio; 5% is allowed."""
    cx, cy, LD = 58, 42, np.longdouble
    KE, corner = fem.element_stiffness(0.3).astype(LD), ((0, 0), (0, 1), (1, 1), (1, 0))
    parts = {}
    for a, b in ((0, 0), (0, 1), (1, 0), (1, 1)):  # P^T KE P of the four children of a coarse element
        P = np.zeros((8, 8), LD)
        for n, (r, c) in enumerate(corner):
            s, t = LD(b + c) / 2, LD(a + r) / 2
            for d in range(2):
                P[2 * n + d, d::2] = (1 - s) * (1 - t), s * (1 - t), s * t, (1 - s) * t
        parts[a, b] = P.T @ KE @ P
    x = soft_design(2 * cx, 2 * cy, "block") * np.random.default_rng(1).uniform(0.5, 1.0, (2 * cy, 2 * cx))
    E = x[0].astype(LD) + np.ldexp(x[1].astype(LD), -k)
    K = sum(E[a::2, b::2, None, None] * parts[a, b] for a, b in parts)

    def rows(K, v):
        ve = np.concatenate([v[r:r + cy, c:c + cx] for r, c in corner], axis=2)
        f, out = (K * ve[:, :, None]).sum(-1), np.zeros(v.shape, LD)
        for n, (r, c) in enumerate(corner):
            out[r:r + cy, c:c + cx] += f[..., 2 * n:2 * n + 2]
        return out

    m = mto.Mesh(2 * cx, 2 * cy, n_coarsen=1)
    for l in range(-1, 2):
        m.set_launch_shape(l, warps)
    m.set_design(dev(x), [1.0, 2.0 ** -k], 1.0)
    total = []
    for seed in range(6):
        v = np.random.default_rng(seed).uniform(-1, 1, (cy + 1, cx + 1, 2))
        v[0] = 0.0
        y = m.apply_operator(0, dev(v)).cpu().numpy().astype(LD)
        err = (y - rows(K, v.astype(LD))) / rows(abs(K), abs(v).astype(LD))
        total.append((err[12:31, 16:43].astype(float) ** 2).mean())  # the block's nodes
    assert np.mean(total) ** 0.5 <= 1.05 * 9.2e-17
    m.close()


@pytest.mark.parametrize("power", [-960, 0, 1000])
@pytest.mark.parametrize("warps", [MARCH, ROWS])
def test_void_block_at_extreme_sizes(mto, warps, power):
    """The usual void beside solids, values near both ends of float64, each row by its own terms."""
    nx, ny = 40, 22
    x = dirichlet_design(nx, ny, 4, seed=4)
    x[:, 5:9, 3:30] = 0.0
    x[3, 5:9, 3:30] = 1.0
    Es = [1.0, 0.5, 0.25, 1e-9]
    lv = multigrid.build_hierarchy(nx, ny, fem.simp_moduli(x, Es, 3.0), fem.element_stiffness(0.3), BOTTOM, 1)
    m = build(mto, nx, ny, 1, x, Es, warps=warps)
    for l in range(2):
        v = np.random.default_rng(l).standard_normal(m.level_shape(l))
        check_rows(m, lv, l, v, 2.0 ** power)  # a power of two: exact in the reference too
    m.close()


@pytest.mark.parametrize("ratio", [1e-9, 1e-12, 1e-24])
def test_soft_parts_of_a_large_mesh(mto, ratio):
    """Marching tasks in full blocks on the finest grid, tiles below it, soft patches of several sizes.
    Here a cycle in float64 instructions throughout is within 1.0e-13 of the oracle's (on the stiff nodes
    4.1e-11, also at ratio 1: the large smooth response to a random residual), so 20 times that is allowed."""
    nx, ny, nc, fixed = 512, 480, 5, BOTTOM
    x = np.zeros((2, ny, nx))
    for j, i, h, w in ((30, 40, 3, 5), (100, 200, 17, 31), (250, 20, 64, 130), (301, 300, 150, 90), (470, 500, 10, 12)):
        x[1, j:j + h, i:i + w] = 1.0
    x[0] = 1.0 - x[1]
    Es = [1.0, ratio]
    lv = multigrid.build_hierarchy(nx, ny, fem.simp_moduli(x, Es, 3.0), fem.element_stiffness(0.3), fixed, nc)
    m = build(mto, nx, ny, nc, x, Es, fixed)
    rng = np.random.default_rng(6)
    for l in (nc, nc - 1):
        v = rng.choice([-1.0, 1.0], m.level_shape(l)) * rng.uniform(0.5, 1.0, m.level_shape(l))
        check_rows(m, lv, l, v * 2.0 ** rng.integers(-20, 21, v.shape[:2] + (1,)))
    r = rng.standard_normal((ny + 1, nx + 1, 2))
    r[0] = 0.0
    z = m.apply_preconditioner(dev(r)).cpu().numpy().ravel()[lv[nc].free]
    ref = multigrid.vcycle_preconditioner(lv, 0.6, 2, 2)(r.ravel()[lv[nc].free])
    assert np.linalg.norm(z - ref) <= 2e-12 * np.linalg.norm(ref)
    stiff = lv[nc].diag > 0.1
    assert np.linalg.norm((z - ref)[stiff]) <= 8e-10 * np.linalg.norm(ref[stiff])
    m.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("at", [(3, 5), (20, 31), (23, 44)])
@pytest.mark.parametrize("power", [50, 100, 900])
def test_one_large_value(mto, power, at, warps, prec):
    """A spike does not reach beyond its neighbours' rows (K p's operator in both precisions)."""
    nx, ny = 44, 24
    x, Es = dirichlet_design(nx, ny, 2, seed=3), [1.0, 0.3]
    lv = multigrid.build_hierarchy(nx, ny, fem.simp_moduli(x, Es, 3.0), fem.element_stiffness(0.3), BOTTOM, 1)
    m = build(mto, nx, ny, 1, x, Es, warps=warps, precision=prec)
    v = np.ones((ny + 1, nx + 1, 2))
    v[at] = 2.0 ** power
    check_rows(m, lv, 1, v)
    v = np.random.default_rng(power).standard_normal(v.shape)
    v[at] = (2.0 ** power, -0.75 * 2.0 ** power)
    check_rows(m, lv, 1, v)
    m.close()


@pytest.mark.parametrize("opts", [dict(), dict(nu2=1), dict(flexible=1, rr_every=3)])
@pytest.mark.parametrize("warps", [MARCH, ROWS])
@pytest.mark.parametrize("kind", ["block", "quadrant"])
@pytest.mark.parametrize("ratio", [1e-9, 1e-15, 1e-21, 1e-27, 1e-30])
def test_solve_with_soft_parts(mto, ratio, kind, warps, opts):
    """Converges as the oracle's float64 iteration does."""
    nx = ny = 32
    x, Es, f = soft_design(nx, ny, kind), [1.0, ratio], load_top_edge(nx, ny)
    m = build(mto, nx, ny, 2, x, Es, warps=warps, tol=1e-8, max_it=60, **opts)
    u, st = m.solve(dev(f))
    ref = solver.solve_pcgmg(nx, ny, x, Es, 3.0, f, n_coarsen=2, tol=1e-8, max_it=60, **opts)
    assert ref["converged"] and abs(st["iters"] - ref["iters"]) <= 1
    assert solver.true_relative_residual(nx, ny, fem.simp_moduli(x, Es, 3.0), f, u.cpu().numpy()) <= 2e-8
    m.close()
