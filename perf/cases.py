"""What is measured: the work a program has this library do, through its public entry points.

Five kinds of pass, each a call (or the calls of one step) that a program makes:

  solve   one structure: lambda and u of every occurrence (fetirp_solve_device), with the pattern factorisation
          (fetirp_factorize) in front of it where "factor" is set, which is a whole time-to-solution step
  apply   the block interface operator Q = P^T F P V (fetirp_apply_block_device), the call of a program that runs
          its own Krylov iteration
  split   the same operator on the split of one interface vector (fetirp_apply_split_device)
  factor  registering a pattern: its factorisation and its operators S^+ and N read back (fetirp_get_pattern)
  serve   a handful of requests of uneven structures through a server over a resident pattern library

Meshes, layouts and sizes come from fetirp_gen (the configurations of the tests and the benchmark); the topology
of a case is fixed, the loads and the vectors come from the seed.  exact() restates every pass with torch in FP64
from the assembled stiffness matrices, the links and the coordinates alone.
"""
from __future__ import annotations

import functools
import weakref

import numpy as np
import torch

import fetirp_gen as gen
import paper_1208_6387_gb300.fetirp as F
from fetirp_gen.configs import batched_uneven, elastic_grid, fill_structure, heat_grid
from fetirp_gen.layout import set_nodal_load

HISTORY = 16 << 30   # cap of the direction history of a solve (a state then fits the card several times)


# --------------------------------------------------------------------------------------------------- the cases
def _case(name, kind, physics, m, grid, k, precision, **more):
    c = {"name": name, "kind": kind, "physics": physics, "m": m, "gx": grid[0], "gy": grid[1],
         "gz": grid[2] if len(grid) > 2 else 1, "k": k, "precision": precision, "patterns": 1, "checker": False,
         "rotate": physics == "elastic", "factor": False,
         "tol": 1e-11 if physics == "heat" else 1e-10 if m <= 8 else 2e-10, "precond": "identity", "iterations": 0, "requests": 0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest structure anyone solves: 2D heat, 2 x 2 occurrences of an 8 x 8 pattern; launches and latency
        _case("solve_heat8_2x2_fp64", "solve", "heat", 8, (2, 2), 4, "fp64", iterations=6),
        # the benchmark's 2D heat step: factorisation and solve on a 1 / 1000 checkerboard of 64 occurrences
        _case("step_heat32_8x8_auto", "solve", "heat", 32, (8, 8), 8, "auto", checker=True, factor=True, tol=5e-13,
              iterations=650),
        # the benchmark's default step: three 16^3 elastic patterns, 192 rotated occurrences; the largest case
        _case("step_elastic16_192_bf16x3", "solve", "elastic", 16, (4, 6, 8), 4, "bf16x3", patterns=3, factor=True,
              iterations=175),
        # a batch of uneven elastic blocks (6^3, 8^3, 12^3) solved together at the automatic precision
        _case("step_batch24_auto", "solve", "batch", 12, (24, 1), 12, "auto", factor=True, rotate=False,
              iterations=100),
        # a mid-size elastic structure whose factors are resident, FP32 products inside the FP64 refinement
        _case("solve_elastic8_27_fp32", "solve", "elastic", 8, (3, 3, 3), 9, "fp32", iterations=90),
        # registering an elastic pattern: factorisation, S^+ and the rigid modes back on the host
        _case("factor_elastic12", "factor", "elastic", 12, (1, 1, 1), 1, "fp64"),
        # F-applies of the large elastic structure: plain FP64, and the mixed form the benchmark's solve uses
        _case("apply_elastic16_192_fp64_k4", "apply", "elastic", 16, (4, 6, 8), 4, "fp64", patterns=3),
        _case("apply_elastic16_192_bf16x3_k4", "apply", "elastic", 16, (4, 6, 8), 4, "bf16x3", patterns=3),
        # a wide block on a mid-size structure (the default block width)
        _case("apply_elastic12_64_tf32x3_k32", "apply", "elastic", 12, (4, 4, 4), 32, "tf32x3"),
        # a ragged one: odd pattern size, odd layout, odd width, FP32 products
        _case("apply_elastic7_30_fp32_k5", "apply", "elastic", 7, (2, 3, 5), 5, "fp32", patterns=2),
        # the sparse-column form on the medium structure of the tests
        _case("split_elastic8_48_tf32x3_k30", "split", "elastic", 8, (3, 4, 4), 30, "tf32x3", patterns=3),
        # six requests of uneven structures, served concurrently from a resident library
        _case("serve_6_requests_auto", "serve", "library", 16, (1, 1), 8, "auto", requests=6, iterations=60),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _elastic_m(rng, hi):
    """An elastic pattern size; on 13^3 a rigid-mode pivot sits at the zero-pivot threshold, so it is left out."""
    m = _log_int(rng, 3, hi)
    return 12 if m == 13 else m


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "apply", "split", "factor", "serve"])
    physics = rng.choice(["heat", "elastic", "elastic"])
    k = _log_int(rng, 1, 32)
    if kind == "serve":
        return _drop(_case("", "serve", "library", 16, (1, 1), _log_int(rng, 2, 16), rng.choice(["auto", "fp32"]),
                           requests=rng.randint(2, 8), iterations=60))
    if kind == "factor":
        m = _log_int(rng, 8, 64) if physics == "heat" else _elastic_m(rng, 15)
        return _drop(_case("", "factor", physics, m, (1, 1, 1), 1, "fp64"))
    if physics == "heat":
        m, grid = _log_int(rng, 6, 64), (rng.randint(2, 9), rng.randint(2, 9))
        precision = rng.choice(["fp64", "fp32", "tf32x3"] if kind != "solve" else ["auto", "fp64", "fp32"])
        precond = rng.choice(["identity", "identity", "dirichlet"]) if kind == "solve" and precision == "fp64" else \
            "identity"
        checker = rng.random() < 0.3 and not (kind == "solve" and precision == "fp64")
        return _drop(_case("", kind, "heat", m, grid, min(k, grid[0] * grid[1]), precision, checker=checker,
                           tol=5e-13 if checker else 1e-11, factor=kind == "solve" and rng.random() < 0.5,
                           precond=precond, iterations=80))
    m = _elastic_m(rng, 14)
    grid = (rng.randint(1, 4), rng.randint(2, 4), rng.randint(1, 5))
    n_occ = grid[0] * grid[1] * grid[2]
    precision = rng.choice(["auto", "fp32", "tf32x3", "bf16x3"] if kind == "solve" else
                           ["fp64", "fp32", "tf32x3"] if kind == "split" else ["fp64", "fp32", "tf32x3", "bf16x3"])
    if kind == "solve" and precision == "fp32":   # the large ones of this form take seconds
        m = min(m, 8)
    return _drop(_case("", kind, "elastic", m, grid, min(k, n_occ), precision, patterns=rng.randint(1, min(3, n_occ)),
                       factor=kind == "solve" and rng.random() < 0.5, iterations=100))


def _drop(c):
    c = dict(c)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------- the inputs
@functools.lru_cache(maxsize=6)
def _topology(physics, m, grid, k, patterns, checker, rotate):
    """The structure without its loads: a fixed seed, so that only the inputs differ between seeds."""
    if physics == "batch":
        return batched_uneven(ms=(6, 8, 12), weights=(0.45, 0.35, 0.2), n_occ=grid[0], seed=0, k_each=max(1, k // 4))
    if physics == "heat":
        return heat_grid(m, grid[:2], kappas=(1.0, 1000.0) if checker else (1.0,), checker=checker, seed=0, k=k)
    return elastic_grid(m, grid, n_patterns=patterns, seed=0, k=k, rotate=rotate)


def _problem(case, seed):
    grid = (case["gx"], case["gy"], case["gz"])
    prob = _topology(case["physics"], case["m"], grid, case["k"], case["patterns"], case["checker"], case["rotate"])
    rng = np.random.default_rng([seed, 1])
    n = prob.n_global_nodes * prob.dpn
    return set_nodal_load(prob, rng.random(n) if prob.dpn == 1 else rng.standard_normal(n))


@functools.lru_cache(maxsize=1)
def _library():
    """Half of the serving library: 2D heat 16^2 and 32^2, 3D elastic 8^3."""
    pats = gen.library_patterns()
    return [pats[0], pats[1], pats[3]]


def _requests(case, seed):
    """Uneven structures of library patterns: their sizes belong to the case, their loads to the seed."""
    pats, out = _library(), []
    for i in range(case["requests"]):
        n_occ = 4 + (37 * i + 11) % 29
        out.append((i % len(pats), fill_structure(pats[i % len(pats)], n_occ, seed=seed * 1009 + i,
                                                  k=min(case["k"], n_occ), rotate=True)))
    return out


def _block(case, prob, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "split":
        return torch.randn(prob.n_lambda, generator=g, device="cuda", dtype=torch.float64)
    return torch.randn(prob.n_lambda, case["k"], generator=g, device="cuda", dtype=torch.float64)


class _State:
    """A context (and a server) with its buffers; released with the state."""

    def __init__(self, case, ctx):
        self.case, self.ctx, self.srv = case, ctx, None
        self._release = weakref.finalize(self, _State._free, [ctx], [])

    def serve_with(self, srv):
        self.srv = srv
        self._release.detach()
        self._release = weakref.finalize(self, _State._free, [self.ctx], [srv])

    @staticmethod
    def _free(ctxs, srvs):
        for s in srvs:
            F.fetirp_server_destroy(s)
        for c in ctxs:
            F.fetirp_destroy(c)


def prepare(case, seed):
    ctx = F.fetirp_create(F.fetirp_default_options(precision=case["precision"] if case["kind"] == "solve" else "fp64",
                                                   tol=case["tol"], history_bytes=HISTORY))
    st = _State(case, ctx)
    if case["kind"] == "factor":
        pat = _problem(case, seed).patterns[0]
        # another material of the same mesh for every seed
        K = pat.K.tocsr() * (1.0 + np.random.default_rng([seed, 2]).random())
        st.n_dofs = pat.n_dofs
        st.pid = F.fetirp_create_pattern(ctx, pat.n_nodes, pat.dpn, K.indptr, K.indices, K.data, pat.bnd_nodes,
                                         pat.kernel_dim)
        return st
    if case["kind"] == "serve":
        pids = []
        for p in _library():
            K = p.K.tocsr()
            pids.append(F.fetirp_create_pattern(ctx, p.n_nodes, p.dpn, K.indptr, K.indices, K.data, p.bnd_nodes,
                                                p.kernel_dim))
        opts = F.fetirp_default_options(precision=case["precision"], tol=case["tol"], history_bytes=1 << 30)
        st.serve_with(F.fetirp_server_create(ctx, opts, 4, 64 << 30))
        st.requests = [(prob.n_lambda, F.n_u(prob), F.structure_of(prob, {0: pids[li]}))
                       for li, prob in _requests(case, seed)]
        return st
    prob = _problem(case, seed)
    F.load_problem(ctx, prob)
    st.n_lambda = prob.n_lambda
    if case["kind"] == "solve":
        F.fetirp_set_preconditioner(ctx, case["precond"])
        st.c = torch.from_numpy(prob.c).cuda()
        st.lam = torch.empty(prob.n_lambda, dtype=torch.float64, device="cuda")
        st.u = torch.empty(F.n_u(prob), dtype=torch.float64, device="cuda")
    else:
        F.fetirp_prepare(ctx, prob.n_lambda, prob.c)
        st.v = _block(case, prob, seed)
        st.q = torch.empty(prob.n_lambda, case["k"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()   # the library runs on its own stream
    return st


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "apply":
        F.fetirp_apply_block_device(st.ctx, case["k"], st.v.data_ptr(), st.q.data_ptr(),
                                    F.PRECISIONS[case["precision"]])
        return {"q": st.q}
    if kind == "split":
        F.fetirp_apply_split_device(st.ctx, st.v.data_ptr(), st.q.data_ptr(), F.PRECISIONS[case["precision"]])
        return {"q": st.q}
    if kind == "solve":
        if case["factor"]:
            F.fetirp_factorize(st.ctx)
        F.fetirp_solve_device(st.ctx, st.n_lambda, st.c.data_ptr(), st.lam.data_ptr(), st.u.data_ptr())
        return {"lambda": st.lam, "u": st.u}
    if kind == "factor":
        F.fetirp_factorize(st.ctx)
        _, _, S, N = F.fetirp_get_pattern(st.ctx, st.pid, st.n_dofs)
        return {"splus": S, "kernel": N}
    tickets = [F.fetirp_server_submit(st.srv, s) for _, _, s in st.requests]
    out = {}
    for i, (t, (nl, nu, _)) in enumerate(zip(tickets, st.requests)):
        out["lambda%d" % i], out["u%d" % i] = F.fetirp_server_wait(st.srv, t, nl, nu)[:2]
    return out


# --------------------------------------------------------------------------------------------------- the work
def _factor_work(pat):
    """Flops of a pattern's set-up: the banded factorisation of the interior and its coupling to the trace, the
    Schur complement's factor and the inverse of its square."""
    dim = pat.dim
    band = (pat.m - 1) ** (dim - 1) * pat.dpn
    n_i, n_b = pat.n_dofs - pat.n_b, pat.n_b
    return n_i * band ** 2 + 2.0 * n_i * band * n_b + n_b ** 3


def _apply_work(prob, k, es):
    """Bytes and flops of one block F-apply: the vectors, every pattern's operator once, the local products."""
    by, fl = 16.0 * prob.n_lambda * k, 0.0
    for i, p in enumerate(prob.patterns):
        n = sum(o.pattern == i for o in prob.occs)
        by += es * p.n_b ** 2
        fl += 2.0 * p.n_b ** 2 * n * k
    return by, fl


def work(case):
    es = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "serve":
        by = fl = 0.0
        for _, prob in _requests(case, 0):
            b, f = _apply_work(prob, prob.k, 4)
            by += 8.0 * (2 * F.n_u(prob) + 2 * prob.n_lambda) + b
            fl += case["iterations"] * f
        return {"bytes": by, "flops": fl}
    prob = _problem(case, 0)
    if case["kind"] == "factor":
        p = prob.patterns[0]
        return {"bytes": 12.0 * p.K.nnz + 8.0 * p.n_b ** 2 + 8.0 * p.n_dofs * p.kernel_dim, "flops": _factor_work(p)}
    by, fl = _apply_work(prob, case["k"] if case["kind"] != "split" else 1, es)
    if case["kind"] == "split":
        by += 8.0 * prob.n_lambda * case["k"]
    if case["kind"] == "solve":
        by += 8.0 * (2 * F.n_u(prob) + 2 * prob.n_lambda)
        fl *= case["iterations"]
        if case["factor"]:
            fl += sum(_factor_work(p) for p in prob.patterns)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------------- the same in plain FP64
def _rigid(prob, pat):
    """Kernel of a pattern from its coordinates: constants (heat), translations and rotations (elasticity)."""
    x = torch.from_numpy(pat.coords - pat.coords.mean(0)).cuda()
    if pat.dpn == 1:
        return torch.ones(len(x), 1, dtype=torch.float64, device="cuda")
    N = torch.zeros(len(x), 3, 6, dtype=torch.float64, device="cuda")
    for c in range(3):
        N[:, c, c] = 1.0
        a, b = (c + 1) % 3, (c + 2) % 3
        N[:, a, 3 + c], N[:, b, 3 + c] = -x[:, b], x[:, a]
    return N.reshape(-1, 6)


def _condense(pat, scale=1.0):
    """Boundary and interior dofs, the interior Cholesky factor, K_ib and the Schur complement."""
    K = torch.from_numpy((pat.K * scale).toarray()).cuda()
    dof = np.arange(pat.dpn)
    b = (pat.bnd_nodes.astype(np.int64)[:, None] * pat.dpn + dof).ravel()
    i = np.setdiff1d(np.arange(pat.n_dofs), b)
    b, i = torch.from_numpy(b).cuda(), torch.from_numpy(i).cuda()
    Kib = K[i][:, b]
    Li = torch.linalg.cholesky(K[i][:, i])
    W = torch.linalg.solve_triangular(Li, Kib, upper=False)
    S = K[b][:, b] - W.T @ W
    return b, i, Li, Kib, 0.5 * (S + S.T)


def _schur_pinv(pat, S, b, prob):
    Nb, _ = torch.linalg.qr(_rigid(prob, pat)[b])
    a = S.diagonal().mean()
    X = torch.cholesky_inverse(torch.linalg.cholesky(S + a * Nb @ Nb.T)) - (Nb @ Nb.T) / a
    return 0.5 * (X + X.T)


def _links(prob):
    """Per occurrence: multiplier rows, their positions (boundary node, component) and signs."""
    out = []
    for o in prob.occs:
        pat = prob.patterns[o.pattern]
        pos = np.full(pat.n_nodes, -1, dtype=np.int64)
        pos[pat.bnd_nodes] = np.arange(len(pat.bnd_nodes))
        at = pos[o.link_local_node] * prob.dpn + o.link_global_comp.astype(np.int64)
        out.append((torch.from_numpy(o.link_lambda_row.astype(np.int64)).cuda(), torch.from_numpy(at).cuda(),
                    torch.from_numpy(o.link_sign.astype(np.float64)).cuda()))
    return out


def _turn(prob, o, X, back):
    """Vectors of an occurrence's nodes (dofs x columns) from the pattern frame to the global one, or back."""
    if prob.dpn == 1:
        return X
    R = torch.from_numpy(np.asarray(prob.occs[o].rot, dtype=np.float64)[:prob.dpn, :prob.dpn]).cuda()
    return torch.einsum("cd,ndk->nck", R.T if back else R, X.reshape(-1, prob.dpn, X.shape[1])).reshape(X.shape)


def _exact_apply(prob, V):
    """P^T F P V by its definition, with the Moore-Penrose inverse of every pattern's Schur complement."""
    pinv, modes, seen = [], [], {}
    for p in prob.patterns:
        key = (p.m, p.dpn, float(p.K.data[0]))
        if key not in seen:
            b, _, _, _, S = _condense(p)
            seen[key] = (_schur_pinv(p, S, b, prob), _rigid(prob, p)[b])
        pinv.append(seen[key][0])
        modes.append(seen[key][1])
    links = _links(prob)
    kd = modes[0].shape[1]
    G = torch.zeros(prob.n_lambda, kd * prob.n_occ, dtype=torch.float64, device="cuda")
    for o, (rows, at, sg) in enumerate(links):
        Ng = _turn(prob, o, modes[prob.occs[o].pattern], False)
        G[rows, kd * o:kd * (o + 1)] += sg[:, None] * Ng[at]
    C = torch.linalg.cholesky(G.T @ G)

    def P(X):
        for _ in range(2):
            X = X - G @ torch.cholesky_solve(G.T @ X, C)
        return X

    X = P(V)
    Q = torch.zeros_like(X)
    for o, (rows, at, sg) in enumerate(links):
        p = prob.occs[o].pattern
        y = torch.zeros(prob.patterns[p].n_b, X.shape[1], dtype=torch.float64, device="cuda")
        y.index_add_(0, at, sg[:, None] * X[rows])
        z = _turn(prob, o, pinv[p] @ _turn(prob, o, y, True), False)
        Q.index_add_(0, rows, sg[:, None] * z[at])
    return P(Q)


def _split_of(prob, r):
    """Column g: the share of r on the rows of the occurrences of group g."""
    V = torch.zeros(prob.n_lambda, prob.k, dtype=torch.float64, device="cuda")
    n = torch.zeros(prob.n_lambda, dtype=torch.float64, device="cuda")
    for o, (rows, _, _) in enumerate(_links(prob)):
        V[:, int(prob.groups[o])].index_add_(0, rows, torch.ones(len(rows), dtype=torch.float64, device="cuda"))
        n.index_add_(0, rows, torch.ones(len(rows), dtype=torch.float64, device="cuda"))
    return V * (r / n)[:, None]


def _exact_solve(prob):
    """u from the assembled interface problem (every interior condensed), lambda from the occurrences'
    equilibria B^T lambda = f - K u: node by node, B B^T lambda = B (f - K u)."""
    dpn = prob.dpn
    used = np.unique(np.concatenate([o.node_map[prob.patterns[o.pattern].bnd_nodes] for o in prob.occs]))
    n = len(used) * dpn
    if n > 20000:
        return None
    slot = np.full(prob.n_global_nodes, -1, dtype=np.int64)
    slot[used] = np.arange(len(used))
    cond = [_condense(p) for p in prob.patterns]
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    g = torch.zeros(n, 1, dtype=torch.float64, device="cuda")
    loads, where, schur = [], [], []
    for o, occ in enumerate(prob.occs):
        b, i, Li, Kib, S = cond[occ.pattern]
        f = _turn(prob, o, torch.from_numpy(occ.f_global).cuda()[:, None], True)
        gl = f[b] - Kib.T @ torch.cholesky_solve(f[i], Li)
        at = torch.from_numpy((slot[occ.node_map[prob.patterns[occ.pattern].bnd_nodes]][:, None] * dpn +
                               np.arange(dpn)).ravel()).cuda()
        Sg = _turn(prob, o, _turn(prob, o, S, False).T.contiguous(), False)
        A[at[:, None], at[None, :]] += Sg
        g[at] += _turn(prob, o, gl, False)
        loads.append((f, _turn(prob, o, gl, False)))
        where.append(at)
        schur.append(Sg)
    fixed = torch.from_numpy((slot[prob.dirichlet_nodes][:, None] * dpn + np.arange(dpn)).ravel()).cuda()
    ub = torch.zeros(n, 1, dtype=torch.float64, device="cuda")
    ub[fixed, 0] = torch.from_numpy(prob.dirichlet_values.ravel().copy()).cuda()
    free = torch.ones(n, dtype=torch.bool, device="cuda")
    free[fixed] = False
    fr = torch.nonzero(free)[:, 0]
    Af = A[fr][:, fr]
    C = torch.linalg.cholesky(Af)
    rhs = g[fr] - A[fr][:, fixed] @ ub[fixed]
    x = torch.cholesky_solve(rhs, C)
    for _ in range(2):
        x = x + torch.cholesky_solve(rhs - Af @ x, C)
    ub[fr] = x
    us, rho = [], torch.zeros(prob.n_lambda, dtype=torch.float64, device="cuda")
    rows2 = torch.full((prob.n_lambda, 2), -1, dtype=torch.int64, device="cuda")
    sign2 = torch.zeros(prob.n_lambda, 2, dtype=torch.float64, device="cuda")
    dof = torch.zeros(prob.n_lambda, dtype=torch.int64, device="cuda")
    for o, (rows, at, sg) in enumerate(_links(prob)):
        occ = prob.occs[o]
        b, i, Li, Kib, _ = cond[occ.pattern]
        f, gg = loads[o]
        ug = ub[where[o]]
        res = gg - schur[o] @ ug
        rho.index_add_(0, rows, sg * res[at, 0])
        e = (rows2[rows, 0] >= 0).long()
        rows2[rows, e], sign2[rows, e], dof[rows] = o, sg, where[o][at]
        ul = torch.zeros(prob.patterns[occ.pattern].n_dofs, 1, dtype=torch.float64, device="cuda")
        ul[b] = _turn(prob, o, ug, True)
        ul[i] = torch.cholesky_solve(f[i] - Kib @ ul[b], Li)
        us.append(_turn(prob, o, ul, False)[:, 0])
    lam = torch.zeros(prob.n_lambda, dtype=torch.float64, device="cuda")
    order = torch.argsort(dof, stable=True)
    _, counts = torch.unique_consecutive(dof[order], return_counts=True)
    starts = torch.cumsum(counts, 0) - counts
    for c in torch.unique(counts).tolist():
        idx = order[starts[counts == c][:, None] + torch.arange(c, device="cuda")]
        oc, sg = rows2[idx], sign2[idx]
        same = (oc[:, :, None, :, None] == oc[:, None, :, None, :]) & (oc[:, :, None, :, None] >= 0)
        BBt = (same * (sg[:, :, None, :, None] * sg[:, None, :, None, :])).sum((-1, -2))
        lam[idx] = torch.linalg.solve(BBt, rho[idx])
    return lam, torch.cat(us)


def _exact_factor(prob, seed):
    """S^+ and N of the zero-pivot factorisation, interior dofs first and the trace last: the dropped dofs are the
    last ones on which the kernel is independent."""
    pat = prob.patterns[0]
    b, i, _, _, S = _condense(pat, 1.0 + np.random.default_rng([seed, 2]).random())
    N = _rigid(prob, pat)
    Nb = N[b].cpu().numpy()
    z, basis = [], np.zeros((0, Nb.shape[1]))
    for j in range(len(Nb) - 1, -1, -1):
        v = Nb[j] - basis.T @ (basis @ Nb[j])
        v = v - basis.T @ (basis @ v)
        if np.linalg.norm(v) > 1e-7 * np.linalg.norm(Nb[j]) and len(z) < Nb.shape[1]:
            z.append(j)
            basis = np.vstack([basis, v / np.linalg.norm(v)])
    z = sorted(z)
    r = torch.from_numpy(np.setdiff1d(np.arange(len(Nb)), z)).cuda()
    Sp = torch.zeros_like(S)
    Sp[r[:, None], r[None, :]] = torch.cholesky_inverse(torch.linalg.cholesky(S[r][:, r]))
    return {"splus": Sp, "kernel": N @ torch.linalg.inv(N[b][z])}


def exact(case, seed):
    if case["kind"] == "serve":
        out = {}
        for n, (_, prob) in enumerate(_requests(case, seed)):
            out["lambda%d" % n], out["u%d" % n] = _exact_solve(prob) or (None, None)
        return out
    prob = _problem(case, seed)
    if case["kind"] == "factor":
        return _exact_factor(prob, seed)
    if case["kind"] == "apply":
        return {"q": _exact_apply(prob, _block(case, prob, seed))}
    if case["kind"] == "split":
        return {"q": _exact_apply(prob, _split_of(prob, _block(case, prob, seed)))}
    got = _exact_solve(prob)
    return None if got is None else {"lambda": got[0], "u": got[1]}
