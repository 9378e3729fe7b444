"""What a user of the P_k auxiliary-space solver has it do, as measurable cases.

A case names a kind of call, a degree k, a mesh size n (n^3 cubes of 6 tetrahedra) and the
options in use. Kinds:
  solve    one load, Problem.solve on a problem that is set up (CG, or FGMRES with the
           multiplicative form where "krylov" says so)
  block    several loads in one Problem.solve
  adjoint  one step of a coefficient fit: autograd.solve and the gradient of a misfit, with
           the operator re-assembled and the preconditioner rebuilt for the step's kappa
  spmv, smoother, prec, vcycle   one application of that operator, as a caller's own Krylov
           method would use it
  stokes   Problem.stokes_solve (Taylor-Hood)
Inputs are jittered meshes of the unit cube, coefficients that are 1 or lognormal per
element, smooth loads for single solves and N(0,1) entries for blocks and operators.
"""
import itertools
import math

import numpy as np
import torch

# nominal entries per row of an interior mesh, and CG iterations to 1e-8 with kappa = 1
_ROW = {1: 15.0, 2: 28.1, 3: 46.6, 4: 73.6}
_ITERS = {1: 15, 2: 22, 3: 36, 4: 46}


def _case(name, kind, k, n, lognormal=False, fp32=False, level="jacobi", krylov="cg", ncols=1):
    c = dict(kind=kind, k=k, n=n, lognormal=lognormal, fp32=fp32, level=level, krylov=krylov, ncols=ncols)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small model problem with every option left at its default: latency of one solve
        _case("solve_p2_n8", "solve", 2, 8, level="gs"),
        # the ordinary FP64 solve, coefficient 1
        _case("solve_p3_n32", "solve", 3, 32),
        # heterogeneous medium in FP64, long rows
        _case("solve_p4_n24_lognormal", "solve", 4, 24, lognormal=True),
        # the largest single solve: 7 million unknowns, FP32 preconditioner
        _case("mixed_p4_n48_lognormal", "solve", 4, 48, lognormal=True, fp32=True),
        # an odd mesh with the FP32 preconditioner and Gauss-Seidel on every level
        _case("mixed_p2_n33", "solve", 2, 33, fp32=True, level="gs"),
        # the paper's outer method: FGMRES around the multiplicative form
        _case("fgmres_p3_n16", "solve", 3, 16, krylov="fgmres"),
        # 3 velocity components times 16 loads at once
        _case("block_p2_n40_c48", "block", 2, 40, fp32=True, ncols=48),
        # a handful of loads on a small odd mesh: a padded block
        _case("block_p3_n9_c5", "block", 3, 9, lognormal=True, ncols=5),
        # one gradient step of a coefficient fit, setup included
        _case("adjoint_p3_n24", "adjoint", 3, 24, lognormal=True, fp32=True),
        # one application of the preconditioner inside a caller's own method
        _case("prec_p4_n32", "prec", 4, 32, lognormal=True),
        # one small product with the operator
        _case("spmv_p2_n21", "spmv", 2, 21),
        # Stokes flow, Taylor-Hood P2-P1
        _case("stokes_p2_n12", "stokes", 2, 12),
    ]


_MOST = {1: 64, 2: 48, 3: 32, 4: 24}


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["block"] * 3 + ["adjoint"] * 2 + ["spmv", "smoother", "prec", "prec", "vcycle"] + ["stokes"])
    k = rng.choice([1, 2, 2, 3, 3, 4, 4])
    if kind == "stokes":
        k = rng.choice([2, 2, 3])
    most = _MOST[k]
    if kind in ("block", "adjoint"):
        most = most * 2 // 3
    if kind == "stokes":
        most = 16 if k == 2 else 8
    n = int(round(math.exp(rng.uniform(math.log(4), math.log(most)))))
    krylov = "fgmres" if kind == "solve" and rng.random() < 0.15 else "cg"
    # a preconditioner in FP32 is used inside a solve; an operator is applied alone in FP64
    fp32 = kind in ("solve", "block", "adjoint") and krylov == "cg" and rng.random() < 0.5
    ncols = rng.randint(2, 48) if kind == "block" else 1
    return _case(None, kind, k, n, rng.random() < 0.5, fp32, rng.choice(["jacobi", "gs"]), krylov, ncols)


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _mesh(n, seed):
    """n^3 cubes of 6 tetrahedra; interior vertices moved by at most 0.15 / n per
    coordinate, which keeps every tetrahedron positively oriented."""
    m = n + 1
    ijk = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    inside = ((ijk > 0) & (ijk < n)).all(1)
    xyz = ijk / n
    xyz[inside] += (np.random.default_rng(seed).random((int(inside.sum()), 3)) - 0.5) * (0.3 / n)
    c = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)
    tets = np.empty((n**3, 6, 4), np.int32)
    for s, p in enumerate(itertools.permutations(range(3))):
        at, path = np.zeros(3, int), [np.zeros(3, int)]
        for axis in p:
            at = at + np.eye(3, dtype=int)[axis]
            path.append(at)
        if s in (1, 2, 5):  # odd permutations
            path[2], path[3] = path[3], path[2]
        for a in range(4):
            v = c + path[a]
            tets[:, s, a] = (v[:, 0] * m + v[:, 1]) * m + v[:, 2]
    return xyz, tets.reshape(-1, 4)


def _kappa(case, nt, seed):
    return np.exp(np.random.default_rng([seed, 1]).standard_normal(nt)) if case["lognormal"] else np.ones(nt)


def _smooth(x, n, seed, stream):
    """A smooth load (or field) at the points x: four random products of sines, times h^3."""
    r = np.random.default_rng([seed, stream])
    f = np.zeros(len(x))
    for _ in range(4):
        q = r.integers(1, 4, 3)
        f += r.standard_normal() * np.prod(np.sin(np.pi * q * x), axis=1)
    return f / n**3


def _noise(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _options(case):
    o = dict(level_smoother=1 if case["level"] == "jacobi" else 0, precond_precision=1 if case["fp32"] else 0)
    if case["krylov"] == "fgmres":
        o.update(krylov=1, mode=1)
    return o


def prepare(case, seed):
    from paper_1204_2586_gb300 import Problem

    xyz, tets = _mesh(case["n"], seed)
    kappa = _kappa(case, len(tets), seed)
    P = Problem(xyz, tets, case["k"], kappa)
    s = dict(kind=case["kind"], P=P, options=_options(case))
    if case["kind"] != "adjoint":
        P.setup(**s["options"])
    kind = case["kind"]
    if kind in ("solve", "adjoint"):
        x = P.dofmap()[1]
        s["b"] = torch.tensor(_smooth(x, case["n"], seed, 2), device="cuda")
    if kind == "adjoint":
        s["b"].requires_grad_(True)
        s["kappa"] = torch.tensor(kappa, device="cuda", requires_grad=True)
        s["seen"] = torch.tensor(_smooth(x, case["n"], seed, 3), device="cuda")
    elif kind == "block":
        s["b"] = _noise((P.nh, case["ncols"]), seed)
    elif kind in ("spmv", "smoother", "prec"):
        s["b"] = _noise(P.nh, seed)
    elif kind == "vcycle":
        s["b"] = _noise(P.nH, seed)
    elif kind == "stokes":
        P.stokes_setup()
        s["b"] = torch.cat([_noise(3 * P.stokes_nh, seed), torch.zeros(P.stokes_np, dtype=torch.float64, device="cuda")])
    return s


def run(s):
    P, kind, b = s["P"], s["kind"], s["b"]
    if kind in ("solve", "block"):
        return P.solve(b)[0]
    if kind == "adjoint":
        from paper_1204_2586_gb300 import autograd

        u = autograd.solve(s["kappa"], b, P, **s["options"])
        loss = 0.5 * ((u - s["seen"]) ** 2).sum()
        dkappa, db = torch.autograd.grad(loss, (s["kappa"], b))
        return {"u": u.detach(), "dkappa": dkappa, "db": db}
    if kind == "spmv":
        return P.spmv(b)
    if kind == "smoother":
        return P.apply_smoother(b)
    if kind == "prec":
        return P.apply_prec(b)
    if kind == "vcycle":
        return P.apply_vcycle(b)
    return P.stokes_solve(b)[0]


def work(case):
    """Each pass over the operator (one for the product, one for the sweep, per iteration:
    12 bytes an entry, 8 in the sweep in FP32) and the vectors that an iteration reads and
    writes; two operations an entry. Iterations are nominal."""
    k, n, cols, kind = case["k"], case["n"], case["ncols"], case["kind"]
    nh = float(k * n - 1) ** 3
    nnz = _ROW[k] * nh
    coarse = 15.0 * float(n - 1) ** 3
    sweep = nnz * (8 if case["fp32"] else 12) + 24 * nh
    product = nnz * 12 + 16 * nh
    cycle = 3 * coarse * (8 if case["fp32"] else 12)
    if kind == "spmv":
        return {"bytes": product, "flops": 2 * nnz}
    if kind == "smoother":
        return {"bytes": sweep, "flops": 2 * nnz}
    if kind == "vcycle":
        return {"bytes": cycle, "flops": 6 * coarse}
    if kind == "prec":
        return {"bytes": sweep + cycle + 32 * nh, "flops": 2 * nnz + 6 * coarse}
    iters = _ITERS[k] * (1.6 if case["lognormal"] else 1.0)
    passes = 2.0
    if case["krylov"] == "fgmres":
        iters, passes = 0.7 * iters, 5.0
    if kind == "stokes":
        iters, cols = 60.0, 3
    one = {"bytes": product + sweep + (passes - 2) * product + cycle + 80 * nh * cols, "flops": 2 * (passes * nnz + 3 * coarse) * cols}
    times = iters * (2 if kind == "adjoint" else 1)
    return {"bytes": times * one["bytes"], "flops": times * one["flops"]}


# ---------------------------------------------------------------------------------------
# the same in 64 bits: element matrices from closed-form integrals, conjugate gradients
# ---------------------------------------------------------------------------------------
def _multi(k, d, least=0):
    return [m for m in itertools.product(range(least, k + 1), repeat=d) if sum(m) == k]


def _stiffness_tables(k):
    """S[a, b, m, n] = (1/|T|) int (d phi_m / d l_a)(d phi_n / d l_b), phi_m = 1 at node m."""
    mons = _multi(k, 4)
    nodes = np.array(mons) / k
    coef = np.linalg.inv(np.array([[np.prod(x ** np.array(a)) for a in mons] for x in nodes]))  # [monomial, node]

    def integral(a):
        return 6.0 * math.prod(math.factorial(v) for v in a) / math.factorial(sum(a) + 3)

    S = np.zeros((4, 4, len(mons), len(mons)))
    for a, b in itertools.product(range(4), repeat=2):
        G = np.zeros((len(mons), len(mons)))
        for i, p in enumerate(mons):
            for j, q in enumerate(mons):
                if p[a] and q[b]:
                    t = [u + v for u, v in zip(p, q)]
                    t[a] -= 1
                    t[b] -= 1
                    G[i, j] = p[a] * q[b] * integral(t)
        S[a, b] = coef.T @ G @ coef
    return S


def _unknowns(xyz, tets, k):
    """(element to unknown, -1 on the boundary; coordinates of the unknowns): vertices, then
    edges, faces and elements, each in the order of their sorted vertices."""
    nv, nt, mons = len(xyz), len(tets), _multi(k, 4)
    t = tets.astype(np.int64)
    order = np.argsort(t, axis=1)
    rank = np.argsort(order, axis=1)  # place of local vertex a among the element's sorted ones
    faces = [np.sort(np.delete(t, o, 1), axis=1) for o in range(4)]
    fkey = np.stack([(f[:, 0] * nv + f[:, 1]) * nv + f[:, 2] for f in faces], 1)
    fids, finv, fcount = np.unique(fkey.ravel(), return_inverse=True, return_counts=True)
    finv = finv.reshape(nt, 4)
    pairs = list(itertools.combinations(range(4), 2))
    ekey = np.stack([np.minimum(t[:, a], t[:, b]) * nv + np.maximum(t[:, a], t[:, b]) for a, b in pairs], 1)
    eids, einv = np.unique(ekey.ravel(), return_inverse=True)
    einv = einv.reshape(nt, 6)
    outer = fcount[finv] == 1
    vb, eb = np.zeros(nv, bool), np.zeros(len(eids), bool)
    for o in range(4):
        on = outer[:, o]
        for a in range(4):
            if a != o:
                vb[t[on, a]] = True
        for e, (a, b) in enumerate(pairs):
            if o not in (a, b):
                eb[einv[on, e]] = True
    per_e, per_f, per_i = k - 1, (k - 1) * (k - 2) // 2, (k - 1) * (k - 2) * (k - 3) // 6
    off_e = nv
    off_f = off_e + len(eids) * per_e
    off_i = off_f + len(fids) * per_f
    edge_of = {p: e for e, p in enumerate(pairs)}
    face_rank = {m: r for r, m in enumerate(_multi(k, 3, 1))}
    elem_rank = {m: r for r, m in enumerate(_multi(k, 4, 1))}
    node = np.empty((nt, len(mons)), np.int64)
    for m, mi in enumerate(mons):
        on = [a for a in range(4) if mi[a]]
        if len(on) == 1:
            node[:, m] = t[:, on[0]]
        elif len(on) == 2:
            a, b = on
            node[:, m] = off_e + einv[:, edge_of[a, b]] * per_e + np.where(t[:, a] > t[:, b], mi[a], mi[b]) - 1
        else:
            table = face_rank if len(on) == 3 else elem_rank
            base = off_f + finv[:, [a for a in range(4) if not mi[a]][0]] * per_f if len(on) == 3 else off_i + np.arange(nt) * per_i
            place = np.zeros(nt, np.int64)
            r = rank[:, on]
            for perm in itertools.permutations(range(len(on))):
                rows = (np.argsort(r, axis=1) == np.array(perm)).all(1)
                place[rows] = table[tuple(mi[on[q]] for q in perm)]
            node[:, m] = base + place
    edge = np.zeros(off_i + nt * per_i, bool)
    edge[:nv] = vb
    edge[off_e:off_f] = np.repeat(eb, per_e)
    edge[off_f:off_i] = np.repeat(fcount == 1, per_f)
    number = np.cumsum(~edge) - 1
    number[edge] = -1
    dof = number[node]
    x = np.zeros((int((~edge).sum()), 3))
    for m, mi in enumerate(mons):
        rows = dof[:, m] >= 0
        x[dof[rows, m]] = np.einsum("a,tac->tc", np.array(mi) / k, xyz[t[rows]])
    return dof, x


def _element_factors(xyz, tets):
    """|T| grad l_a . grad l_b, [elements, 16]"""
    x = torch.tensor(xyz[tets], device="cuda")
    J = (x[:, 1:] - x[:, :1]).transpose(1, 2)
    g = torch.linalg.inv(J)
    g = torch.cat([-g.sum(1, keepdim=True), g], 1)
    return ((g @ g.transpose(1, 2)) * (torch.linalg.det(J) / 6.0)[:, None, None]).reshape(len(tets), 16)


def _cg(A, b, diag):
    """Columns of A x = b by conjugate gradients with the diagonal, to the rounding of 64 bits."""
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag[:, None]
    p, rho, goal = z.clone(), (r * z).sum(0), 1e-14 * b.norm(dim=0)
    for i in range(20000):
        q = A @ p
        a = rho / (p * q).sum(0)
        x += a * p
        r -= a * q
        if i % 20 == 0 and bool((r.norm(dim=0) <= goal).all()):
            break
        z = r / diag[:, None]
        new = (r * z).sum(0)
        p = z + (new / rho) * p
        rho = new
    return x


def exact(case, seed):
    kind, k, n = case["kind"], case["k"], case["n"]
    if kind not in ("solve", "block", "adjoint", "spmv"):
        return None  # sweeps in the solver's own colour order, cycles of its own hierarchy, saddle point
    xyz, tets = _mesh(n, seed)
    dof, x = _unknowns(xyz, tets, k)
    nh, nl = len(x), dof.shape[1]
    kappa = torch.tensor(_kappa(case, len(tets), seed), device="cuda")
    S = torch.tensor(_stiffness_tables(k), device="cuda").reshape(16, nl * nl)
    factors = _element_factors(xyz, tets)
    d = torch.tensor(dof, device="cuda")
    rows, cols = d[:, :, None].expand(-1, nl, nl).reshape(-1), d[:, None, :].expand(-1, nl, nl).reshape(-1)
    keep = (rows >= 0) & (cols >= 0)
    values = ((factors * kappa[:, None]) @ S).reshape(-1)[keep]
    A = torch.sparse_coo_tensor(torch.stack([rows[keep], cols[keep]]), values, (nh, nh))
    del rows, cols, keep, values
    A = A.coalesce()
    i, j = A.indices()
    diag = torch.zeros(nh, dtype=torch.float64, device="cuda")
    diag[i[i == j]] = A.values()[i == j]
    del i, j
    A = A.to_sparse_csr()
    if kind == "spmv":
        return A @ _noise(nh, seed)
    if kind == "block":
        return _cg(A, _noise((nh, case["ncols"]), seed), diag)
    u = _cg(A, torch.tensor(_smooth(x, n, seed, 2), device="cuda")[:, None], diag)
    if kind == "solve":
        return u[:, 0]
    lam = _cg(A, u - torch.tensor(_smooth(x, n, seed, 3), device="cuda")[:, None], diag)
    inside = (d >= 0).double()
    ue, le = (v[d.clamp(min=0), 0] * inside for v in (u, lam))
    dkappa = torch.zeros(len(tets), dtype=torch.float64, device="cuda")
    for ab in range(16):
        dkappa -= factors[:, ab] * ((le @ S[ab].reshape(nl, nl)) * ue).sum(1)
    return {"u": u[:, 0], "dkappa": dkappa, "db": lam[:, 0]}
