"""Performance cases of the framework: what its users have it do, over the range of sizes they do it at.

Every case goes through the public entry points (Mesh, Batch, Poisson,
compliance) with new inputs made on the GPU from a seed.  Kinds:

  solve     one design: operators, PCG solve, compliance and sensitivities
            (one call of a design study; with warm=True one step of the
            optimiser's loop, started from the previous design's solution)
  grad      compliance as a torch autograd function, forward and backward
            (a design driven by a torch optimiser)
  host      the same as solve from pinned host memory, through the pipelined
            host call (a caller that keeps its design on the host)
  batch     independent problems of uneven mesh size with two load cases each,
            one launch (a study over many designs)
  vcycle    the multigrid preconditioner alone (a caller with its own Krylov
            method)
  operator  the stiffness operator alone on the finest grid (the same)
  poisson   the scalar Poisson solver, one or many right-hand sides
"""

import math

import numpy as np
import torch

import paper_2301_07457_gb300 as mto

NU = 0.3
DEV = "cuda"
BOTTOM, LEFT, RIGHT = mto.EDGE_BOTTOM, mto.EDGE_LEFT, mto.EDGE_RIGHT
# Solid moduli by number of phases; the last phase of each is void.
MODULI = {2: [1.0, 1e-9], 4: [1.0, 0.5, 0.25, 1e-9], 5: [1.0, 0.7, 0.5, 0.3, 0.15]}


def listed():
    return [
        # The smallest mesh of the benchmark's workloads: launches and latency.
        dict(name="solve_64_fp64", kind="solve", nx=64, ny=64, nc=2, precision="fp64", tol=1e-10,
             phases=4, edges=BOTTOM, rhs=1, design="dirichlet", warm=False),
        # One step of the optimisation loop of the mesh sweep, in its middle range.
        dict(name="loop_256_fp64", kind="solve", nx=256, ny=256, nc=4, precision="fp64", tol=1e-8,
             phases=4, edges=BOTTOM, rhs=1, design="smooth", warm=True),
        # A ragged wall clamped on two edges, two load cases at once.
        dict(name="ragged_200x136_mixed", kind="solve", nx=200, ny=136, nc=3, precision="mixed", tol=1e-8,
             phases=4, edges=BOTTOM | LEFT, rhs=2, design="dirichlet", warm=False),
        # The differentiable workload: five solid phases, forward and backward.
        dict(name="grad_512_fp64", kind="grad", nx=512, ny=512, nc=5, precision="fp64", tol=1e-8,
             phases=5, edges=BOTTOM, rhs=1, design="dirichlet"),
        # Pinned host arrays in and out, mixed precision, at the sweep's largest mesh.
        dict(name="host_1024_mixed", kind="host", nx=1024, ny=1024, nc=6, precision="mixed", tol=1e-8,
             phases=4, edges=BOTTOM, rhs=1, design="dirichlet"),
        # The benchmark's headline workload.
        dict(name="solve_2048_mixed", kind="solve", nx=2048, ny=2048, nc=7, precision="mixed", tol=1e-8,
             phases=4, edges=BOTTOM, rhs=1, design="dirichlet", warm=False),
        # The largest float64 solve that the benchmark reports.
        dict(name="solve_4096_fp64", kind="solve", nx=4096, ny=4096, nc=8, precision="fp64", tol=1e-8,
             phases=4, edges=BOTTOM, rhs=1, design="dirichlet", warm=False),
        # A batch of uneven problems, two load cases each, sizes as the batched workload draws them.
        dict(name="batch_8_mixed", kind="batch", sizes="128,256,256,512,512,128,1024,256", precision="mixed",
             tol=1e-8, phases=4),
        # The two building blocks at the headline size.
        dict(name="vcycle_2048_mixed", kind="vcycle", nx=2048, ny=2048, nc=7, precision="mixed", phases=4,
             edges=BOTTOM, design="dirichlet"),
        dict(name="operator_2048_fp64", kind="operator", nx=2048, ny=2048, nc=7, precision="fp64", phases=4,
             edges=BOTTOM, design="dirichlet"),
        # Table 1's problem: one small solve, and many right-hand sides of the largest mesh.
        dict(name="poisson_64", kind="poisson", nx=64, ny=64, nc=5, precision="fp64", tol=1e-8, rhs=1),
        dict(name="poisson_256_x64", kind="poisson", nx=256, ny=256, nc=7, precision="mixed", tol=1e-8, rhs=64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(rng, lo, hi):
    """nelx, nely, coarsenings of a wall of about lo^2..hi^2 elements, seldom a power of two."""
    n = _log(rng, lo, hi)
    aspect = rng.choice([1.0, 1.0, rng.uniform(0.5, 2.0)])
    nc = max(2, min(8, round(math.log2(n / 16.0))))
    return (max(9, round(n * math.sqrt(aspect) / 2 ** nc)) << nc,
            max(9, round(n / math.sqrt(aspect) / 2 ** nc)) << nc, nc)


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "loop", "grad", "host", "batch", "vcycle", "operator", "poisson"])
    precision = rng.choice(["fp64", "mixed"])
    phases = rng.choice([2, 4, 4, 5])
    edges = rng.choice([BOTTOM, BOTTOM, BOTTOM | LEFT, BOTTOM | LEFT | RIGHT])
    design = rng.choice(["dirichlet", "smooth"])
    tol = rng.choice([1e-8, 1e-8, 1e-10])
    if kind in ("solve", "loop"):
        nx, ny, nc = _mesh(rng, 64, 2400)
        return dict(kind="solve", nx=nx, ny=ny, nc=nc, precision=precision, tol=tol, phases=phases, edges=edges,
                    rhs=rng.choice([1, 1, 2]), design=design, warm=kind == "loop")
    if kind == "grad":
        nx, ny, nc = _mesh(rng, 64, 1200)
        return dict(kind=kind, nx=nx, ny=ny, nc=nc, precision=precision, tol=tol, phases=phases, edges=edges,
                    rhs=rng.choice([1, 2]), design=design)
    if kind == "host":
        nx, ny, nc = _mesh(rng, 128, 1500)
        return dict(kind=kind, nx=nx, ny=ny, nc=nc, precision=precision, tol=tol, phases=phases, edges=edges,
                    rhs=1, design=design)
    if kind == "batch":
        sizes = [rng.choice([128, 256, 256, 512, 512, 1024]) for _ in range(rng.randint(3, 10))]
        return dict(kind=kind, sizes=",".join(map(str, sizes)), precision=precision, tol=1e-8, phases=4)
    if kind in ("vcycle", "operator"):
        nx, ny, nc = _mesh(rng, 64, 4096)
        return dict(kind=kind, nx=nx, ny=ny, nc=nc, precision=precision, phases=phases, edges=edges, design=design)
    nc = rng.randint(3, 7)
    return dict(kind="poisson", nx=rng.randint(2, 3) << nc, ny=rng.randint(2, 3) << nc, nc=nc, precision=precision,
                tol=tol, rhs=int(round(_log(rng, 1, 64))))


# -- inputs ------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _design(case, gen, nx, ny):
    """Phase fractions [phases][ny][nx]: Dirichlet(1,..,1) per element, or the
    soft regions of a design half way through an optimisation."""
    P = case["phases"]
    if case.get("design", "dirichlet") == "dirichlet":
        x = torch.empty(P, ny, nx, dtype=torch.float64, device=DEV).exponential_(generator=gen)
        return x / x.sum(0)
    c = torch.randn(P, 5, 5, dtype=torch.float64, device=DEV, generator=gen)
    k = torch.arange(5, dtype=torch.float64, device=DEV)[:, None] * math.pi
    by = torch.cos(k * (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) / ny)
    bx = torch.cos(k * (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) / nx)
    return torch.softmax(1.2 * torch.einsum("pab,ay,bx->pyx", c, by, bx), 0)


def _loads(nx, ny, rhs):
    """Top edge pushed down, right edge pushed sideways."""
    f = torch.zeros(rhs, ny + 1, nx + 1, 2, dtype=torch.float64, device=DEV)
    f[0, ny, :, 1] = -1.0
    if rhs > 1:
        f[1, :, nx, 0] = 1.0
    return f


def _make_mesh(case, nx, ny, nc):
    return mto.Mesh(nx, ny, nu=NU, fixed_edges=case.get("edges", BOTTOM), n_coarsen=nc, precision=case["precision"],
                    tol=case.get("tol", 1e-8))


def _inputs(case, seed):
    """The arrays a case computes with (also those exact() needs)."""
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "poisson":
        return {"f": torch.randn(case["rhs"], case["ny"] + 1, case["nx"] + 1, dtype=torch.float64, device=DEV,
                                 generator=gen)}
    if kind == "batch":
        return [{"x": _design(case, gen, n, n), "f": _loads(n, n, 2), "n": n}
                for n in map(int, case["sizes"].split(","))]
    nx, ny = case["nx"], case["ny"]
    d = {"x": _design(case, gen, nx, ny)}
    if kind in ("vcycle", "operator"):
        d["v"] = torch.randn(ny + 1, nx + 1, 2, dtype=torch.float64, device=DEV, generator=gen)
        return d
    d["f"] = _loads(nx, ny, case["rhs"])
    if case["rhs"] == 1:
        d["f"] = d["f"][0]
    if case.get("warm"):
        # The previous design of the loop: fractions a move of up to 0.2 away.
        d["x_prev"] = 0.9 * d["x"] + 0.1 * _design(case, gen, nx, ny)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "poisson":
        solver = mto.Poisson(case["nx"], case["ny"], n_coarsen=case["nc"], tol=case["tol"],
                             precision=case["precision"])
        return {"kind": kind, "solver": solver, **d}
    E = MODULI[case["phases"]]
    if kind == "batch":
        problems = [{"mesh": _make_mesh(case, p["n"], p["n"], int(math.log2(p["n"])) - 4), "x": p["x"], "E_phase": E,
                     "f": p["f"]} for p in d]
        return {"kind": kind, "batch": mto.Batch(problems)}
    mesh = _make_mesh(case, case["nx"], case["ny"], case["nc"])
    s = {"kind": kind, "mesh": mesh, "E": E, **d}
    if kind == "grad":
        s["x"] = d["x"].requires_grad_(True)
    elif kind == "host":
        s["x"], s["f"] = d["x"].cpu().pin_memory(), d["f"].cpu().pin_memory()
    elif kind in ("vcycle", "operator"):
        mesh.set_design(d["x"], E, 3.0)
    elif case.get("warm"):
        mesh.set_design(d["x_prev"], E, 3.0)
        s["u0"], _ = mesh.solve(d["f"])
    return s


def run(state):
    kind = state["kind"]
    if kind == "solve":
        mesh = state["mesh"]
        mesh.set_design(state["x"], state["E"], 3.0)
        u, _ = mesh.solve(state["f"], u0=state.get("u0"))
        C, g = mesh.compliance_grad(state["f"], u)
        return {"u": u, "C": C, "dcdx": g}
    if kind == "grad":
        C = mto.compliance(state["x"], state["mesh"], state["f"], state["E"], 3.0)
        (g,) = torch.autograd.grad(C, state["x"])
        return {"C": C.detach(), "dcdx": g}
    if kind == "host":
        state["mesh"].run_host_async(state["x"], state["E"], 3.0, state["f"])
        u, C, g, _ = state["mesh"].run_host_wait()
        return {"u": u, "C": C, "dcdx": g}
    if kind == "batch":
        batch = state["batch"]
        for p in batch.problems:  # a cold start in each pass
            p["u"].zero_()
        batch.run()
        return [{"u": p["u"], "C": p["compliance"], "dcdx": p["dcdx"]} for p in batch.problems]
    if kind == "vcycle":
        return state["mesh"].apply_preconditioner(state["v"])
    if kind == "operator":
        return state["mesh"].apply_operator(state["mesh"].opts.n_coarsen, state["v"])
    u, _ = state["solver"].solve(state["f"])
    return u


# Arithmetic of one PCG iteration per finest node (outer operator and vector
# updates about 50, the V-cycle's sweeps about 200 over all grids), and the
# iterations that these solves take.
ITERATION_FLOPS, ITERATIONS = 250, 26
POISSON_FLOPS, POISSON_ITERATIONS = 90, 6


def work(case):
    kind = case["kind"]
    if kind == "poisson":
        nodes = (case["nx"] + 1) * (case["ny"] + 1) * case["rhs"]
        return {"bytes": 16.0 * nodes, "flops": float(POISSON_FLOPS * POISSON_ITERATIONS * nodes)}
    if kind == "batch":
        parts = [dict(kind="solve", nx=n, ny=n, phases=case["phases"], rhs=2) for n in map(int, case["sizes"].split(","))]
        every = [work(p) for p in parts]
        return {k: sum(w[k] for w in every) for k in ("bytes", "flops")}
    nodes, elements = (case["nx"] + 1) * (case["ny"] + 1), case["nx"] * case["ny"]
    if kind == "vcycle":
        return {"bytes": 32.0 * nodes + 8.0 * elements, "flops": 200.0 * nodes}
    if kind == "operator":
        return {"bytes": 32.0 * nodes + 8.0 * elements, "flops": 36.0 * nodes}
    out = 0 if kind == "grad" else 16
    return {"bytes": (16.0 + out) * nodes * case["rhs"] + 16.0 * elements * case["phases"],
            "flops": float(ITERATION_FLOPS * ITERATIONS * nodes * case["rhs"])}


# -- the same in plain float64 torch -----------------------------------------
def _element_matrix():
    """The 8 x 8 plane-stress matrix of a unit-square Q4 element (2 x 2 Gauss points)."""
    c = 1.0 / (1.0 - NU * NU)
    D = np.array([[c, c * NU, 0], [c * NU, c, 0], [0, 0, c * (1 - NU) / 2]])
    K = np.zeros((8, 8))
    for gx in (-1, 1):
        for gy in (-1, 1):
            a, b = gx / math.sqrt(3.0), gy / math.sqrt(3.0)
            dx = np.array([-(1 - b), 1 - b, 1 + b, -(1 + b)]) / 2
            dy = np.array([-(1 - a), -(1 + a), 1 + a, 1 - a]) / 2
            B = np.zeros((3, 8))
            B[0, 0::2], B[1, 1::2], B[2, 0::2], B[2, 1::2] = dx, dy, dy, dx
            K += B.T @ D @ B / 4
    return torch.tensor(K, device=DEV)


CORNERS = ((0, 0), (0, 1), (1, 1), (1, 0))  # (row, column) of the nodes BL, BR, TR, TL


def _free(nx, ny, edges):
    m = torch.ones(ny + 1, nx + 1, 1, dtype=torch.float64, device=DEV)
    if edges & BOTTOM:
        m[0] = 0
    if edges & LEFT:
        m[:, 0] = 0
    if edges & RIGHT:
        m[:, nx] = 0
    return m


def _gather(v, ny, nx):
    return torch.cat([v[..., r:r + ny, c:c + nx, :] for r, c in CORNERS], -1)


def _scatter(q, ny, nx):
    out = torch.zeros(ny + 1, nx + 1, 2, dtype=torch.float64, device=DEV)
    for n, (r, c) in enumerate(CORNERS):
        out[r:r + ny, c:c + nx] += q[..., 2 * n:2 * n + 2]
    return out


def _direct(E, f, edges):
    """u = K^-1 f by block Cholesky over the node rows; f [rhs][ny+1][nx+1][2]."""
    ny, nx = E.shape
    KE, m = _element_matrix(), 2 * (nx + 1)
    free = _free(nx, ny, edges).expand(ny + 1, nx + 1, 2).reshape(ny + 1, m)
    cols = 2 * torch.arange(nx, device=DEV)

    def block(rows, columns, row):
        """Entries of element row `row` between the nodes of two of its node rows."""
        B = torch.zeros(m * m, dtype=torch.float64, device=DEV)
        for a in rows:
            for b in columns:
                for i in range(2):
                    for k in range(2):
                        at = (cols + 2 * CORNERS[a][1] + i) * m + cols + 2 * CORNERS[b][1] + k
                        B.index_add_(0, at, E[row] * KE[2 * a + i, 2 * b + k])
        return B.view(m, m)

    low, high = (0, 1), (3, 2)
    chol, link, W, y = [], [], None, []
    g = (f.reshape(f.shape[0], ny + 1, m) * free).permute(1, 2, 0)
    for j in range(ny + 1):
        S = torch.zeros(m, m, dtype=torch.float64, device=DEV)
        if j < ny:
            S += block(low, low, j)
        if j > 0:
            S += block(high, high, j - 1)
        S = S * free[j][:, None] * free[j] + torch.diag(1 - free[j])
        r = g[j]
        if j > 0:
            S -= W.T @ W
            r = r - W.T @ y[-1]
        L = torch.linalg.cholesky(S)
        chol.append(L)
        y.append(torch.linalg.solve_triangular(L, r, upper=False))
        if j < ny:
            B = block(high, low, j) * free[j + 1][:, None] * free[j]
            W = torch.linalg.solve_triangular(L, B.T, upper=False)
            link.append(W)
    u = torch.zeros_like(g)
    for j in range(ny, -1, -1):
        r = y[j] if j == ny else y[j] - link[j] @ u[j + 1]
        u[j] = torch.linalg.solve_triangular(chol[j].T, r, upper=True)
    return u.permute(2, 0, 1).reshape(f.shape)


def _moduli(x, Es):
    return sum(x[i] ** 3 * e for i, e in enumerate(Es))


def _exact_solve(x, Es, f, edges):
    ny, nx = x.shape[1:]
    fb = f.reshape(-1, ny + 1, nx + 1, 2)
    u = _direct(_moduli(x, Es), fb, edges)
    ue = _gather(u, ny, nx)
    ue = ue - ue[..., :2].repeat(1, 1, 1, 4)  # K_e ignores translations
    energy = ((ue @ _element_matrix()) * ue).sum(-1).sum(0)
    g = torch.stack([-3.0 * x[i] ** 2 * e * energy for i, e in enumerate(Es)])
    return {"u": u.reshape(f.shape), "C": (fb * u).sum((1, 2, 3)), "dcdx": g}


def _exact_vcycle(case, E, r):
    """One V(2,2) cycle of damped Jacobi (0.6) with Galerkin coarse grids and a dense coarsest solve."""
    nx, ny, edges = case["nx"], case["ny"], case["edges"]
    # Coarse element matrices: sums over the four children of Q^T K_child Q.
    Qs = {}
    for a in (0, 1):
        for b in (0, 1):
            Q = torch.zeros(8, 8, dtype=torch.float64, device=DEV)
            for n, (rr, cc) in enumerate(CORNERS):
                s, t = (b + cc) / 2, (a + rr) / 2
                for k, w in enumerate(((1 - s) * (1 - t), s * (1 - t), s * t, (1 - s) * t)):
                    Q[2 * n, 2 * k] = Q[2 * n + 1, 2 * k + 1] = w
            Qs[a, b] = Q
    K = [E[..., None, None] * _element_matrix()]
    for _ in range(case["nc"]):
        K.append(sum(Q.T @ K[-1][a::2, b::2] @ Q for (a, b), Q in Qs.items()))
    masks = [_free(nx >> l, ny >> l, edges) for l in range(case["nc"] + 1)]

    def apply(l, v):
        k = K[l]
        return masks[l] * _scatter((k @ _gather(v * masks[l], *k.shape[:2])[..., None])[..., 0], *k.shape[:2])

    def up(v):  # bilinear interpolation
        h, w = v.shape[:2]
        o = torch.zeros(2 * h - 1, 2 * w - 1, 2, dtype=torch.float64, device=DEV)
        o[::2, ::2] = v
        o[::2, 1::2] = (v[:, 1:] + v[:, :-1]) / 2
        o[1::2] = (o[2::2] + o[:-1:2]) / 2
        return o

    def down(v):  # its transpose
        h = v[::2].clone()
        h[1:] += v[1::2] / 2
        h[:-1] += v[1::2] / 2
        o = h[:, ::2].clone()
        o[:, 1:] += h[:, 1::2] / 2
        o[:, :-1] += h[:, 1::2] / 2
        return o

    def cycle(l, b):
        k, m = K[l], masks[l]
        h, w = k.shape[:2]
        if l == case["nc"]:
            node = torch.arange((h + 1) * (w + 1), device=DEV).view(h + 1, w + 1)
            dof = torch.cat([torch.stack([2 * node[i:i + h, c:c + w], 2 * node[i:i + h, c:c + w] + 1], -1)
                             for i, c in CORNERS], -1).view(-1, 8)
            n = 2 * node.numel()
            A = torch.zeros(n * n, dtype=torch.float64, device=DEV)
            A.index_add_(0, (dof[:, :, None] * n + dof[:, None, :]).reshape(-1), k.reshape(-1))
            keep = torch.nonzero(m.expand(-1, -1, 2).reshape(-1) > 0)[:, 0]
            z = torch.zeros(n, dtype=torch.float64, device=DEV)
            z[keep] = torch.linalg.solve(A.view(n, n)[keep][:, keep], b.reshape(-1)[keep])
            return z.view(h + 1, w + 1, 2)
        diag = _scatter(torch.diagonal(k, dim1=-2, dim2=-1), h, w)
        wd = 0.6 * m / diag
        z = wd * b
        z = z + wd * (b - apply(l, z))
        z = z + m * up(cycle(l + 1, masks[l + 1] * down(m * (b - apply(l, z)))))
        for _ in range(2):
            z = z + wd * (b - apply(l, z))
        return z

    return cycle(0, masks[0] * r)


def exact(case, seed):
    kind = case["kind"]
    d = _inputs(case, seed)
    if kind == "poisson":
        def sines(n):
            k = torch.arange(1, n, dtype=torch.float64, device=DEV)
            return torch.sin(math.pi * k[:, None] * k / n) * math.sqrt(2.0 / n), torch.cos(math.pi * k / n)
        (Sx, cx), (Sy, cy) = sines(case["nx"]), sines(case["ny"])
        lam = (8 - 2 * cx[None] - 2 * cy[:, None] - 4 * cx[None] * cy[:, None]) / 3
        u = torch.zeros_like(d["f"])
        u[:, 1:-1, 1:-1] = Sy @ ((Sy @ d["f"][:, 1:-1, 1:-1] @ Sx) / lam) @ Sx
        return u
    Es = MODULI[case["phases"]]
    if kind == "batch":  # the direct solve of a 1024^2 wall takes too long
        none = {"u": None, "C": None, "dcdx": None}
        return [_exact_solve(p["x"], Es, p["f"], BOTTOM) if p["n"] <= 256 else none for p in d]
    nx, ny = case["nx"], case["ny"]
    if kind == "operator":
        m = _free(nx, ny, case["edges"])
        return m * _scatter(_moduli(d["x"], Es)[..., None] * (_gather(m * d["v"], ny, nx) @ _element_matrix()), ny, nx)
    if kind == "vcycle":
        if nx * ny > 5e6:
            return None
        E = _moduli(d["x"], Es)
        if case["precision"] == "mixed":  # whose V-cycle has bfloat16 moduli
            E = E.to(torch.bfloat16).to(torch.float64)
        return _exact_vcycle(case, E, d["v"])
    if nx * ny > 3e5:
        return None
    got = _exact_solve(d["x"].detach(), Es, d["f"], case["edges"])
    if kind == "grad":
        return {"C": got["C"].sum(), "dcdx": got["dcdx"]}
    return got
