"""The work a program has this library do, as cases that can be timed and checked.

A case is one call sequence of a user's program: the mesh stands, new data
arrives, the solver runs, the solution (and gradients) come back.  `prepare`
makes what such a program holds before the call (tree or forest, source,
boundary values, coefficient, target), `run` is the call, `exact` its answer
as plain torch gives it in 64 bits: the composite system of the leaves (or,
on a uniform grid, its sine transform), assembled and solved here.

Meshes, sources and sizes are those of the paper's tests (arXiv:1701.04329
Sec. 4) and of the batched and differentiable workloads of
paper_1701_04329_gb300/workloads.py; every solve goes to the library's default
tolerance, 1e-10 of the source's largest value.
"""
import math

import numpy as np
import torch

from paper_1701_04329_gb300 import afgpu
from paper_1701_04329_gb300.autograd import PoissonSolve

DEV = "cuda"
F64 = torch.float64
DIR, NEU, PER = afgpu.AFG_BC_DIRICHLET, afgpu.AFG_BC_NEUMANN, afgpu.AFG_BC_PERIODIC

# sides: boundary types of -x,+x,-y,+y[,-z,+z], one letter each
LETTER = {"d": DIR, "n": NEU, "p": PER}


def _case(name, kind, dim, box, uniform, extra, **kw):
    c = dict(kind=kind, dim=dim, box=box, uniform=uniform, extra=extra, precision="fp64", sides="d" * (2 * dim),
             rx=1, ry=1, rz=1, op=0, prolong=0, sources=1, width=0.04, trees=1)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one small 2D problem (64^2 cells, three levels around a Gaussian): the paper's first test;
        # what a 2D simulation solves every time step
        _case("quadtree_small_fp64", "solve", 2, 8, 4, 3),
        # the same kind of step on a 3 x 2 block of root boxes periodic across: a channel
        _case("quadtree_channel_mixed", "solve", 2, 8, 3, 3, precision="mixed", sides="ddpp", rx=3, ry=2, sources=3,
              width=0.08),
        # the 3D octree of 17.6 million unknowns around two small sources, plain and mixed: the large production solve
        _case("octree_sources_fp64", "solve", 3, 8, 6, 2, sources=2, width=0.01),
        _case("octree_sources_mixed", "solve", 3, 8, 6, 2, precision="mixed", sources=2, width=0.01),
        # the paper's scaling problem: a uniform 512^3 grid
        _case("uniform_512_mixed", "uniform", 3, 8, 7, 0, precision="mixed"),
        # differentiable solve, forward and backward: gradient of a misfit with respect to source and boundary data
        _case("blobs_gradient_fp64", "grad", 3, 8, 5, 1, sources=8, width=0.03),
        _case("blobs_gradient_mixed", "grad", 3, 8, 5, 1, precision="mixed", sources=8, width=0.03),
        # a batch of independent quadtrees of uneven depth (levels 4 to 9), one call for all of them
        _case("forest_mixed", "forest", 2, 8, 3, 6, precision="mixed", trees=128),
        # a few shallow trees in plain FP64: a small ensemble
        _case("forest_small_fp64", "forest", 2, 16, 2, 2, trees=12),
        # a dielectric jump of 100 in a quarter of the domain, 256^2 and refined: the paper's second test
        _case("jump_2d_fp64", "solve", 2, 8, 6, 1, op=1, sources=2, width=0.05),
        # the same operator in cylindrical coordinates (axisymmetric discharge), mixed precision, 16^2 boxes
        _case("jump_rz_mixed", "solve", 2, 16, 5, 2, op=2, precision="mixed", sides="nddd", sources=2, width=0.05),
        # a dielectric jump in 3D, mixed precision
        _case("jump_3d_mixed", "solve", 3, 8, 5, 1, op=1, precision="mixed", sources=2, width=0.04),
    ]


def _cells(c):
    """About how many leaf cells a drawn case has: the uniform grid and, around every source, the finest one."""
    d, reach = c["dim"], 2.5 * c["width"]
    coarse, fine = c["box"] * 2 ** (c["uniform"] - 1), c["box"] * 2 ** (c["uniform"] + c["extra"] - 1)
    part = min(1.0, c["sources"] * (2 * reach + 4 * c["box"] / coarse) ** d) if c["extra"] else 0.0
    return coarse ** d + part * fine ** d


def draw(rng):
    """One more case: sizes over the whole range of the listed ones (the finest uniform level stands for the size,
    a factor 2^dim each), box sizes 8 and 16, sides, blocks of roots, operators and prolongations as they come."""
    kind = rng.choice(["solve2", "solve2", "solve3", "solve3", "grad", "forest", "jump2", "jump3", "uniform"])
    prec = rng.choice(["fp64", "mixed"])
    box = rng.choice([8, 8, 16])
    less = 1 if box == 16 else 0  # the same cells with one level less
    width = round(math.exp(rng.uniform(math.log(0.01), math.log(0.08))), 4)
    n = rng.randint(1, 8)
    pairs = ["dd", "dd", "nd", "dn", "nn", "pp"]
    if kind == "forest":
        return _case(None, "forest", 2, box, 3 - less, rng.randint(0, 6), precision=prec,
                     trees=int(round(math.exp(rng.uniform(math.log(3), math.log(128))))))
    if kind == "uniform":
        return _case(None, "uniform", 3, box, rng.randint(3, 7) - less, 0, precision=prec)
    if kind == "grad":
        c = _case(None, "grad", 3, box, rng.randint(2, 5) - less, rng.randint(0, 1), precision=prec, sources=n,
                  width=width)
    elif kind in ("solve2", "jump2"):
        sides = rng.choice(["dd", "dn", "nd"]) + rng.choice(pairs)
        c = _case(None, "solve", 2, box, rng.randint(2, 7) - less, rng.randint(0, 2), precision=prec, sides=sides,
                  sources=n, width=width)
        if kind == "jump2":  # Dirichlet sides (the axis has none in (r,z)): with more Neumann sides a jump of 100 can stall
            op = rng.choice([1, 2])
            c.update(uniform=min(c["uniform"], 6 - less), op=op, sides="dddd" if op == 1 else "nddd")
        elif rng.random() < 0.3:
            c.update(rx=rng.randint(1, 5), ry=rng.randint(2, 3), uniform=min(c["uniform"], 5))
    else:
        sides = rng.choice(["dd", "dn", "nd"]) + rng.choice(pairs) + rng.choice(pairs)
        c = _case(None, "solve", 3, box, rng.randint(2, 6) - less, rng.randint(0, 2), precision=prec, sides=sides,
                  sources=n, width=width)
        if kind == "jump3":
            c.update(op=1, uniform=min(c["uniform"], 5), extra=min(c["extra"], 1), sides="dd" + sides[4:] + "dd")
        elif rng.random() < 0.25:
            c["prolong"] = rng.choice([1, 2])
            c["uniform"] = min(c["uniform"], 5)
    most = 2e7 if kind in ("solve2", "solve3") else 8e6
    while _cells(c) > most:  # fewer and narrower sources, then less refinement
        if c["sources"] > 1:
            c["sources"] -= 1
        elif c["width"] > 0.01:
            c["width"] = round(max(0.01, 0.7 * c["width"]), 4)
        elif c["extra"]:
            c["extra"] -= 1
        else:
            c["uniform"] -= 1
    return c


# ---- inputs -----------------------------------------------------------------

def _opts(case):
    return afgpu.default_opts(precision=afgpu.AFG_MIXED if case["precision"] == "mixed" else afgpu.AFG_FP64)


def _roots(case):
    return (case["rx"], case["ry"], case["rz"])[: case["dim"]]


def _centres(case, k=0):
    """Where the sources are, in the domain and off its sides: the mesh follows them, so they belong to the case."""
    rng = np.random.default_rng([case["sources"], case["dim"], k])
    return 0.15 + rng.uniform(size=(case["sources"], case["dim"])) * (np.array(_roots(case), dtype=float) - 0.3)


def _source_set(centres, widths, rng):
    """Gaussian sources about the centres (moved by up to a quarter of their width), with amplitudes of either sign."""
    amps = rng.normal(size=len(centres))
    amps += np.where(amps < 0, -0.3, 0.3)
    return centres + 0.25 * widths[:, None] * rng.uniform(-1, 1, size=centres.shape), widths, amps


def _grow(tree, extra, centres, reach):
    """Refines, level by level, the boxes that lie within `reach` of a source (2:1 balance and a two-cell buffer are
    the library's)."""
    N, D = tree.N, tree.D
    for _ in range(extra):
        e = tree.export()
        leaf = e["children"][:, 0] < 0
        lv, idx = e["level"][leaf], e["idx"][leaf]
        size = 2.0 ** (1 - lv)
        lo, hi = (idx - 1) * size[:, None], idx * size[:, None]
        near = np.zeros(len(lv), bool)
        for c, r in zip(centres, reach):
            gap = np.maximum(0.0, np.maximum(lo - c, c - hi))
            near |= (gap ** 2).sum(1) < r * r
        near &= lv == lv.max()
        if not near.any():
            return
        tree.adapt(np.repeat(near.astype(np.int8), N ** D), 2)


def _tree(case, centres, widths, extra=None):
    roots = _roots(case)
    D, extra = case["dim"], case["extra"] if extra is None else extra
    t = afgpu.Tree(D, case["box"], case["uniform"] + extra, roots=None if set(roots) == {1} else roots)
    if set(case["sides"]) != {"d"}:
        t.set_boundary_types([LETTER[s] for s in case["sides"]])
    if case["op"]:
        t.set_operator(case["op"])
    if case["prolong"]:
        t.set_prolongation(case["prolong"])
    t.refine_uniform(case["uniform"])
    _grow(t, extra, centres, (1.5 if case["kind"] == "grad" else 2.5) * widths)
    return t


def _forest(case):
    """The trees of a forest with the centres and widths of their sources: every depth up to the deepest in turn, one
    to four sources each."""
    for k in range(case["trees"]):
        one = dict(case, sources=1 + (k // 3) % 4)
        centres = _centres(one, k)
        widths = 0.01 + 0.07 * np.random.default_rng([k, 1]).uniform(size=len(centres))
        yield _tree(one, centres, widths, 1 + k % case["extra"] if case["extra"] else 0), centres, widths


def _gaussians(x, src):
    out = torch.zeros(len(x), dtype=F64, device=DEV)
    for c, s, a in zip(*src):
        out += a * torch.exp(-((x - torch.tensor(c, dtype=F64, device=DEV)) ** 2).sum(1) / s ** 2)
    return out


def _boundary(case, tree, rng):
    """Smooth data on the domain sides: potentials on Dirichlet sides, outward derivatives on Neumann sides."""
    n = tree.n_bfaces
    if n == 0:
        return torch.zeros(0, dtype=F64, device=DEV)
    x = torch.tensor(tree.face_centers(), device=DEV)
    k = torch.tensor(rng.uniform(1.0, 4.0, size=case["dim"]), dtype=F64, device=DEV)
    return 1e-3 * torch.cos((x * k).sum(1) + rng.uniform(0, 6))


def _eps(x):
    """100 in the lower quarter of every axis, 1 elsewhere."""
    return torch.where((x < 0.25).all(1), 100.0, 1.0).to(F64)


def prepare(case, seed):
    rng = np.random.default_rng([seed, 7])
    opts = _opts(case)
    if case["kind"] == "forest":
        trees, rho = [], []
        for t, centres, widths in _forest(case):
            x = torch.tensor(t.cell_centers(), device=DEV)
            rho.append(_gaussians(x, _source_set(centres, widths, rng)))
            trees.append(t)
        f = afgpu.Forest(trees)
        return dict(kind="forest", forest=f, rho=torch.cat(rho), opts=opts,
                    b=torch.zeros(int(f.faces.sum()), dtype=F64, device=DEV), trees=trees)
    centres, widths = _centres(case), np.full(case["sources"], case["width"])
    t = _tree(case, centres, widths)
    src = _source_set(centres, widths, rng)
    x = t.cell_centers_device()
    st = dict(kind=case["kind"], tree=t, opts=opts, trees=[t])
    if case["kind"] == "uniform":  # constant source of the scaling test, with a little of everything on top
        k = torch.tensor(rng.uniform(1.0, 6.0, size=3), dtype=F64, device=DEV)
        st["rho"] = 1.0 + 0.1 * torch.sin((x * k).sum(1) + rng.uniform(0, 6))
        st["b"] = torch.zeros(t.n_bfaces, dtype=F64, device=DEV)
    else:
        st["rho"] = _gaussians(x, src)
        st["b"] = _boundary(case, t, rng)
    if case["op"]:
        st["eps"] = _eps(x)
        t.set_eps(st["eps"])
    if case["kind"] == "grad":
        other = _source_set(_centres(case, 1), 8 * widths, rng)
        lv = torch.tensor(t.leaf_levels(), device=DEV).repeat_interleave(t.N ** t.D).to(F64)
        st["vol"] = (1.0 / (t.N * 2.0 ** (lv - 1))) ** t.D
        st["target"] = 1e-3 * _gaussians(x, other)
    st["zero"] = torch.zeros_like(st["rho"])
    return st


# ---- one pass ---------------------------------------------------------------

def run(state):
    if state["kind"] == "forest":
        f = state["forest"]
        f.set_rhs(state["rho"])
        f.set_dirichlet(state["b"])
        f.solve(state["opts"])
        return {"u": f.get_solution()}
    t = state["tree"]
    if state["kind"] == "grad":
        rho = state["rho"].detach().requires_grad_(True)
        b = state["b"].detach().requires_grad_(True)
        u = PoissonSolve.apply(rho, b, t, state["opts"])
        loss = 0.5 * (state["vol"] * (u - state["target"]) ** 2).sum()
        loss.backward()
        return {"u": u.detach(), "drho": rho.grad, "db": b.grad}
    t.set_rhs(state["rho"])
    if state["b"].numel():
        t.set_dirichlet(state["b"])
    t.set_solution(state["zero"])
    t.solve(state["opts"])
    return {"u": t.get_solution()}


def _unknowns(case):
    """Leaf cells and boundary faces of the mesh (host work only)."""
    if case["kind"] == "forest":
        trees = [t for t, _, _ in _forest(case)]
    else:
        trees = [_tree(case, _centres(case), np.full(case["sources"], case["width"]))]
    return sum(t.n_leaf_cells for t in trees), sum(t.n_bfaces for t in trees)


def work(case):
    """Bytes: source (and coefficient, target and volumes) and boundary data read once, solution (and gradients)
    written once.  Flops: ten V(2,2) cycles (a factor ten each) of 2D+2 operations per relaxed cell and sweep on
    every level, twice that with the adjoint."""
    cells, faces = _unknowns(case)
    d = case["dim"]
    read = 8 * (cells * (1 + (1 if case["op"] else 0) + (2 if case["kind"] == "grad" else 0)) + faces)
    wrote = 8 * (cells * 2 + faces) if case["kind"] == "grad" else 8 * cells
    flops = 10 * 4 * (2 * d + 2) * cells * 2 ** d / (2 ** d - 1) * (2 if case["kind"] == "grad" else 1)
    return {"bytes": read + wrote, "flops": flops}


# ---- the answer in 64 bits ----------------------------------------------------
# Each leaf cell has one equation, sum over its faces of c (g - u) / h^2 = rho (the mesh is an input, like the
# source: boxes of N^D cells with a level and a position).  g is the value across the face: a leaf cell of the same
# level; the mean of the 2^D finer cells (weighted by r in (r,z)); 2b - u or u + h b at a Dirichlet or Neumann
# side; at a coarser leaf uH/2 + w u - (u_n + u_t [+ u_t'])/4 with w = 1 (2D) or 5/4 (3D), u_n the next cell
# inward, u_t the other cells under the same coarse face.  c is 1, or the harmonic mean of the two cells'
# coefficients (times r_face / r_cell for the r faces).

def _system(case, tree, eps=None):
    """K (n x n, CSR) and B (n x faces, COO) of the leaf equations of one tree, K u + B b = rho."""
    D, N = case["dim"], case["box"]
    roots = _roots(case)
    e = tree.export()
    leaf = e["children"][:, 0] < 0
    lv = torch.tensor(e["level"][leaf].astype(np.int64), device=DEV)
    idx = torch.tensor(e["idx"][leaf].astype(np.int64), device=DEV) - 1
    nl, C = len(lv), N ** D
    loc = torch.stack([(torch.arange(C, device=DEV) // N ** a) % N for a in range(D)], 1)
    pos = (idx[:, None, :] * N + loc[None]).reshape(-1, D)
    lev = lv.repeat_interleave(C)
    n = nl * C
    h = 1.0 / (N * 2.0 ** (lev.to(F64) - 1))
    S = 24 if D == 2 else 19

    def key(l, p):
        k = l.clone()
        for a in range(D):
            k = (k << S) + p[..., a]
        return k

    own = key(lev, pos)
    order = torch.argsort(own)
    own = own[order]

    def find(l, p):
        k = key(l, p)
        at = torch.searchsorted(own, k).clamp(max=n - 1)
        return torch.where(own[at] == k, order[at], -1)

    ar = torch.arange(n, device=DEV)
    one = torch.ones(n, dtype=F64, device=DEV)
    eps = one if eps is None else eps
    rows, cols, vals, brow, bcol, bval = [], [], [], [], [], []
    diag = torch.zeros(n, dtype=F64, device=DEV)

    def put(r, c, v):
        rows.append(r), cols.append(c), vals.append(v)

    # boundary faces: box by box, side by side, first tangential axis fastest
    last = torch.stack([roots[a] * 2 ** (lv - 1) - 1 for a in range(D)], 1)
    kinds = [LETTER[s] for s in case["sides"]]
    out = torch.stack([(idx[:, s // 2] == (0 if s % 2 == 0 else last[:, s // 2])) & (kinds[s] != PER)
                       for s in range(2 * D)], 1)
    F = N ** (D - 1)
    first = ((out.reshape(-1).cumsum(0) - out.reshape(-1).long()) * F).reshape(nl, 2 * D)
    for s in range(2 * D):
        a, up = s // 2, s % 2
        geo = one
        if case["op"] == 2 and a == 0:
            geo = (pos[:, 0] + up).to(F64) / (pos[:, 0].to(F64) + 0.5)
        q = pos.clone()
        q[:, a] += 2 * up - 1
        side = roots[a] * N * 2 ** (lev - 1)
        if kinds[s] == PER:
            q[:, a] %= side
        outside = (q[:, a] < 0) | (q[:, a] >= side)
        w = ar[outside]
        cf = (eps * geo)[w] / h[w] ** 2
        tang = [t for t in range(D) if t != a]
        f = loc[w % C, tang[0]] + (N * loc[w % C, tang[1]] if D == 3 else 0)
        brow.append(w)
        bcol.append(first[w // C, s] + f)
        if kinds[s] == NEU:
            bval.append(cf * h[w])
        else:
            bval.append(2 * cf)
            diag[w] -= 2 * cf
        inside = ~outside
        same = find(lev, q)
        m = inside & (same >= 0)
        w, o = ar[m], same[m]
        cf = 2 * eps[w] * eps[o] / (eps[w] + eps[o]) * geo[w] / h[w] ** 2
        put(w, o, cf)
        diag[w] -= cf
        rest = ar[inside & (same < 0)]
        if not len(rest):
            continue
        up_l, up_p = lev[rest] - 1, q[rest] // 2
        coarse = find(up_l, up_p)
        w, o = rest[coarse >= 0], coarse[coarse >= 0]
        cf = 2 * eps[w] * eps[o] / (eps[w] + eps[o]) * geo[w] / h[w] ** 2
        put(w, o, 0.5 * cf)
        diag[w] += (0.0 if D == 2 else 0.25) * cf
        inward = pos[w].clone()
        inward[:, a] -= 2 * up - 1
        put(w, find(lev[w], inward), -0.25 * cf)
        for t in tang:
            beside = pos[w].clone()
            beside[:, t] ^= 1
            put(w, find(lev[w], beside), -0.25 * cf)
        w = rest[coarse < 0]
        if not len(w):
            continue
        kids, wt = [], []
        for bits in range(2 ** D):
            p = 2 * q[w] + torch.tensor([(bits >> t) & 1 for t in range(D)], device=DEV)
            kids.append(find(lev[w] + 1, p))
            wt.append(p[:, 0].to(F64) + 0.5 if case["op"] == 2 else one[w])
        total = sum(wt)
        ec = sum(x * eps[k] for x, k in zip(wt, kids)) / total
        cf = 2 * eps[w] * ec / (eps[w] + ec) * geo[w] / h[w] ** 2
        for x, k in zip(wt, kids):
            put(w, k, cf * x / total)
        diag[w] -= cf
    put(ar, ar, diag)
    B = (torch.cat(brow), torch.cat(bcol), torch.cat(bval))
    return (torch.cat(rows), torch.cat(cols), torch.cat(vals)), B, n, diag


def _csr(coo, n, transposed=False):
    r, c, v = coo
    if transposed:
        r, c = c, r
    m = torch.sparse_coo_tensor(torch.stack([r, c]), v, (n, n)).coalesce()
    return m.to_sparse_csr()


def _bicgstab(A, diag, b, tol=1e-14, rounds=6, most=6000):
    """A x = b by BiCGStab (van der Vorst 1992) with the diagonal as preconditioner, begun again from the true
    residual until that stops falling."""
    x = torch.zeros_like(b)
    size, best = float(b.norm()), float("inf")
    if size == 0.0:
        return x
    for _ in range(rounds):
        r = b - A @ x
        now = float(r.norm()) / size
        if now < tol or now > 0.5 * best:
            break
        best, stop = now, max(1e-7 * now, 0.3 * tol) * size
        rh, p = r.clone(), r.clone()
        rho, dx = torch.dot(rh, r), torch.zeros_like(b)
        for it in range(most):
            ph = p / diag
            v = A @ ph
            alpha = rho / torch.dot(rh, v)
            s = r - alpha * v
            sh = s / diag
            t = A @ sh
            omega = torch.dot(t, s) / torch.dot(t, t)
            dx += alpha * ph + omega * sh
            r = s - omega * t
            if it % 20 == 19 and float(r.norm()) < stop:
                break
            new = torch.dot(rh, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        x = x + dx if bool(torch.isfinite(dx).all()) else x
    return x


def _sine_solve(case, tree, rho):
    """The uniform grid with u = 0 on its sides: the seven-point system is diagonal in the sine basis."""
    M = case["box"] * 2 ** (case["uniform"] - 1)
    k = torch.arange(1, M + 1, dtype=F64, device=DEV)
    i = torch.arange(M, dtype=F64, device=DEV) + 0.5
    Q = torch.sin(math.pi / M * torch.outer(k, i)) * math.sqrt(2.0 / M)
    Q[-1] /= math.sqrt(2.0)
    lam = -(2 * M * torch.sin(math.pi * k / (2 * M))) ** 2
    e = tree.export()
    N = case["box"]
    idx = torch.tensor(e["idx"][e["children"][:, 0] < 0].astype(np.int64), device=DEV) - 1
    c = torch.arange(N ** 3, device=DEV)
    at = [((idx[:, a] * N)[:, None] + ((c // N ** a) % N)[None]).reshape(-1) for a in range(3)]
    flat = (at[2] * M + at[1]) * M + at[0]
    g = torch.empty(M ** 3, dtype=F64, device=DEV)
    g[flat] = rho
    g = g.reshape(M, M, M)

    def along(m, g):
        for a in range(3):
            g = torch.movedim(torch.tensordot(m, g, dims=([1], [a])), 0, a).contiguous()
        return g

    g = along(Q, g)
    g /= lam[:, None, None] + lam[None, :, None] + lam[None, None, :]
    return along(Q.t().contiguous(), g).reshape(-1)[flat]


def exact(case, seed):
    st = prepare(case, seed)
    rho, b = st["rho"], st["b"]
    if case["kind"] == "uniform":
        return {"u": _sine_solve(case, st["tree"], rho)}
    parts, cell0, face0 = [], 0, 0
    for t in st["trees"]:
        (r, c, v), (br, bc, bv), n, diag = _system(case, t, st.get("eps"))
        parts.append((r + cell0, c + cell0, v, br + cell0, bc + face0, bv, diag))
        cell0 += n
        face0 += t.n_bfaces
    r, c, v, br, bc, bv, diag = (torch.cat(p) for p in zip(*parts))
    K = _csr((r, c, v), cell0)
    rhs = rho.clone()
    if b.numel():
        rhs.index_add_(0, br, -bv * b[bc])
    u = _bicgstab(K, diag, rhs)
    if case["kind"] != "grad":
        return {"u": u}
    del K
    lam = _bicgstab(_csr((r, c, v), cell0, transposed=True), diag, st["vol"] * (u - st["target"]))
    db = torch.zeros_like(b)
    db.index_add_(0, bc, -bv * lam[br])
    return {"u": u, "drho": lam, "db": db}
