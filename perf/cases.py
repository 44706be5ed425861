"""What a user of this library has it do, as cases that can be timed.

A case names a workload and its sizes; ``prepare`` makes the inputs (and the
launch plan a program keeps), ``run`` is one pass through the public entry
points, ``exact`` the same results from plain torch in 64 bits.

Workloads (matrices are column-major and factored in place, so a pass factors
a copy, as a caller that keeps its matrix does):
  lu_solve   calu_factor + calu_getrs: A X = B
  qr_solve   caqr_factor + caqr_geqrs: least squares (or a square system)
  lu, qr     the factorization alone
  tslu, tsqr one tall-skinny panel
  gesv, gels the tensor-core factorization with FP64 refinement
  batch      many uneven CALU and CAQR factorizations in one launch
"""
import math
import os

import torch

import paper_1303_5837_gb300 as ca
from paper_1303_5837_gb300 import tune

DEV = "cuda"
BENCH_TREE = "1024:4f,0f"      # large squares: the benchmark's tree
SERVE_TREE = "256:4b,0b"       # the solve server's defaults
SMALL_TREE = "128:0b"          # 1024 x 1024 configuration
PANEL_TREE = "256:4b,8b,0b"    # tall-skinny panels: four levels
TABLES = {"f64": "tuned_batch_f64.json", "f32": "tuned_batch_f32.json"}


def listed():
    return [
        # the solve server's small end: launches and the host path
        dict(name="lu_solve_96", work="lu_solve", n=96, nrhs=3, b=128, tree=SERVE_TREE, cond=1e2),
        # one mid-size matrix, both factorizations: the panels' column chains
        dict(name="lu_1024", work="lu", m=1024, n=1024, b=64, tree=SMALL_TREE),
        dict(name="qr_1024", work="qr", m=1024, n=1024, b=64, tree=SMALL_TREE),
        # a ragged least-squares request of the server (m = 4 n), few right-hand sides
        dict(name="qr_solve_3001x750", work="qr_solve", m=3001, n=750, nrhs=5, b=128, tree=SERVE_TREE, cond=1e2),
        # tall-skinny panels alone
        dict(name="tslu_1Mx64", work="tslu", m=1048576, n=64, tree=PANEL_TREE),
        dict(name="tsqr_1Mx64", work="tsqr", m=1048576, n=64, tree=PANEL_TREE),
        # large squares in FP64: the trailing updates
        dict(name="lu_solve_10240", work="lu_solve", n=10240, nrhs=1, b=128, tree=BENCH_TREE, cond=1e2),
        dict(name="qr_solve_6144", work="qr_solve", m=6144, n=6144, nrhs=1, b=128, tree=BENCH_TREE, cond=1e2),
        # tensor-core factorization + FP64 refinement, as the server and the benchmark call them
        dict(name="gesv_4096", work="gesv", n=4096, nrhs=1, b=128, tree=BENCH_TREE, cond=1e4, slices=4),
        dict(name="gels_8192x2048", work="gels", m=8192, n=2048, nrhs=4, b=128, tree=SERVE_TREE, cond=1e4, slices=4),
        # the uneven batch (half square, half tall; CALU and CAQR of each), tuned shapes
        dict(name="batch_f64_1024", work="batch", count=1024, shapes=2026, dtype="f64"),
        dict(name="batch_f32_1024", work="batch", count=1024, shapes=2027, dtype="f32"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["lu_solve", "lu", "qr", "qr_solve", "tslu", "tsqr", "gesv", "gels", "batch"])
    cond = 10.0 ** rng.uniform(0.5, 3.0)
    nrhs = rng.randint(1, 16)
    if kind == "lu_solve":
        n = _log_int(rng, 64, 9000)
        return dict(work=kind, n=n, nrhs=nrhs, b=128, tree=BENCH_TREE if n >= 2048 else SERVE_TREE, cond=cond)
    if kind in ("lu", "qr"):
        n = _log_int(rng, 96, 2000)
        m = n + rng.choice([0, 0, rng.randint(1, n)])
        return dict(work=kind, m=m, n=n, b=rng.choice([32, 64]), tree=SMALL_TREE)
    if kind == "qr_solve":
        n = _log_int(rng, 64, 5000)
        m = n if n > 1500 else 4 * n + rng.randint(0, 3)
        return dict(work=kind, m=m, n=n, nrhs=nrhs, b=128, tree=BENCH_TREE if n > 1500 else SERVE_TREE, cond=cond)
    if kind in ("tslu", "tsqr"):
        n = rng.choice([16, 32, 64, rng.randint(8, 64)])
        return dict(work=kind, m=_log_int(rng, 4096, 1 << 20), n=n, tree=PANEL_TREE)
    if kind == "gesv":
        n = _log_int(rng, 256, 4096)
        return dict(work=kind, n=n, nrhs=nrhs, b=128, tree=BENCH_TREE if n >= 2048 else SERVE_TREE,
                    cond=10.0 ** rng.uniform(1.0, 4.0), slices=4)
    if kind == "gels":
        n = _log_int(rng, 128, 2048)
        return dict(work=kind, m=4 * n + rng.randint(0, 3), n=n, nrhs=nrhs, b=128, tree=SERVE_TREE,
                    cond=10.0 ** rng.uniform(1.0, 4.0), slices=4)
    return dict(work=kind, count=_log_int(rng, 64, 1024), shapes=rng.randint(1, 1 << 20), dtype=rng.choice(["f64", "f32"]))


def parse_tree(spec):
    """"<leaf rows>:<fan-in><b|f>,...": binary or flat merges level by level."""
    leaf, levels = spec.split(":")
    return int(leaf), [(int(t[:-1]), ca.BINARY if t[-1] == "b" else ca.FLAT) for t in levels.split(",")]


def make_tree(case):
    leaf, levels = parse_tree(case["tree"])
    if "b" in case:
        leaf = max(leaf, case["b"])
    return ca.make_tree(leaf, levels)


def shape(case):
    return case.get("m", case["n"]), case["n"]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def gaussian(m, n, gen, dtype=torch.float64):
    return torch.randn(n, m, dtype=dtype, device=DEV, generator=gen).t()


def _mix(X, gen):
    """An orthogonal mixing of X's rows: discrete Hartley transform, random
    signs, the transform again (any length, cheap on the device)."""
    n = X.shape[0]
    sign = (torch.randint(0, 2, (n, 1), device=DEV, generator=gen) * 2 - 1).double()
    for k in range(2):
        F = torch.fft.fft(X, dim=0)
        X = (F.real - F.imag) / math.sqrt(n)
        if k == 0:
            X = X * sign
    return X


def conditioned(m, n, cond, gen):
    """U diag(s) V^T, U and V orthogonal, s log-spaced with s_0 / s_(n-1) = cond, in a random order."""
    s = cond ** (-torch.arange(n, dtype=torch.float64, device=DEV) / max(1, n - 1)) * math.sqrt(n)
    X = torch.zeros(m, n, dtype=torch.float64, device=DEV)
    X.diagonal().copy_(s[torch.randperm(n, device=DEV, generator=gen)])
    X = _mix(X, gen)
    X = _mix(X.t().contiguous(), gen)      # n x m: the transposed matrix
    return X.contiguous().t()              # column-major m x n


def batch_layout(case):
    here = os.path.dirname(os.path.abspath(tune.__file__))
    table = tune.load_table(os.path.join(here, TABLES[case["dtype"]]))
    shapes, ops, bs, trees = tune.batch_items(case["shapes"], case["count"], table, 8 if case["dtype"] == "f64" else 4)
    offs, total = [], 0
    for m, n in shapes:
        offs.append(total)
        total += (m * n + 31) // 32 * 32
    return shapes, ops, bs, trees, offs, total


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    kind = case["work"]
    if kind == "batch":
        shapes, ops, bs, trees, offs, total = batch_layout(case)
        dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
        A0 = torch.randn(total, dtype=dtype, device=DEV, generator=gen)
        flat = A0.clone()
        mats = [flat[o: o + m * n].view(n, m).t() for o, (m, n) in zip(offs, shapes)]
        plan = ca.BatchedFactor(mats, ops, bs, [ca.make_tree(L, lv) for L, lv in trees])
        return dict(kind=kind, A0=A0, flat=flat, plan=plan)
    m, n = shape(case)
    A = conditioned(m, n, case["cond"], gen) if "cond" in case else gaussian(m, n, gen)
    s = dict(kind=kind, A=A, tree=make_tree(case), b=case.get("b", n), slices=case.get("slices"))
    if "nrhs" in case:
        B = A @ gaussian(n, case["nrhs"], gen)
        if m > n:  # least squares: right-hand sides outside the range too
            B = B + 0.1 * gaussian(m, case["nrhs"], gen)
        s["B"] = ca.colmajor(B)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "batch":
        s["flat"].copy_(s["A0"])
        s["plan"].run()
        return s["flat"], s["plan"].ipiv_all, s["plan"].qtree_all, s["plan"].info_all
    A, b, tree = s["A"], s["b"], s["tree"]
    if kind == "gesv":
        LU = torch.empty_like(A)
        ipiv = torch.empty(A.shape[1], dtype=torch.int32, device=A.device)
        X, _, _, info = ca.calu_gesv_mixed(A, s["B"], b, tree, slices=s["slices"], exact=True, refine="auto", LU=LU,
                                           ipiv=ipiv)
        return X, LU, ipiv, info
    if kind == "gels":
        QR = torch.empty_like(A)
        X, _, _, info = ca.caqr_gels_mixed(A, s["B"], b, tree, slices=s["slices"], exact=True, QR=QR)
        return X, QR, info
    F = A.clone()
    if kind == "tslu":
        ipiv, info = ca.tslu(F, tree)
        return F, ipiv, info
    if kind == "tsqr":
        qtree, info = ca.tsqr(F, tree)
        return F, qtree, info
    if kind in ("lu", "lu_solve"):
        ipiv, info = ca.calu_factor(F, b, tree)
        if kind == "lu":
            return F, ipiv, info
        X = s["B"].clone()
        ca.calu_getrs(F, ipiv, X)
        return F, ipiv, info, X
    qtree, info = ca.caqr_factor(F, b, tree)
    if kind == "qr":
        return F, qtree, info
    X = s["B"].clone()
    ca.caqr_geqrs(F, b, tree, qtree, X)
    return F, qtree, info, X


def work(case):
    """Standard flop counts; each input read once, each output written once."""
    if case["work"] == "batch":
        shapes, ops, _, _, _, _ = batch_layout(case)
        esz = 8 if case["dtype"] == "f64" else 4
        return {"bytes": float(sum(2 * m * n * esz for m, n in shapes)),
                "flops": float(sum(tune.item_flops(op, m, n) for op, (m, n) in zip(ops, shapes)))}
    m, n = shape(case)
    k, r = min(m, n), case.get("nrhs", 0)
    lu = 2.0 * (m * n * k - (m + n) * k * k / 2.0 + k ** 3 / 3.0)
    qr = 2.0 * m * n * n - 2.0 * n ** 3 / 3.0
    isqr = case["work"] in ("qr", "qr_solve", "tsqr", "gels")
    flops = (qr + (4.0 * m * n - n * n) * r) if isqr else (lu + 2.0 * n * n * r)
    return {"bytes": 8.0 * (2 * m * n + 2 * m * r), "flops": flops}


# ---------------------------------------------------------------------------
# the same results from plain torch in 64 bits
# ---------------------------------------------------------------------------

def rounds(nleaves, levels):
    """Merge rounds of the reduction tree: lists of groups of node indices."""
    out, cur = [], nleaves
    for i, (fan, style) in enumerate(levels):
        f = cur if i == len(levels) - 1 else fan
        sizes = [min(f, cur - s) for s in range(0, cur, f)]
        while max(sizes) > 1:
            groups, at, left = [], 0, []
            for s in sizes:
                w = s if style == ca.FLAT else 2
                cut = [list(range(at + t, at + min(t + w, s))) for t in range(0, s, w)]
                groups += cut
                left.append(len(cut))
                at += s
            out.append(groups)
            sizes = left
        cur = len(sizes)
    return out


def gepp(T):
    """GEPP of a batch of r x c blocks: (factored blocks, row order)."""
    T = T.clone()
    nb, r, c = T.shape
    order = torch.arange(r, device=T.device).repeat(nb, 1)
    at = torch.arange(nb, device=T.device)
    for j in range(min(r, c)):
        p = T[:, j:, j].abs().argmax(dim=1) + j
        row, lab = T[at, p].clone(), order[at, p].clone()
        T[at, p], order[at, p] = T[:, j].clone(), order[:, j].clone()
        T[:, j], order[:, j] = row, lab
        if j + 1 < r:
            T[:, j + 1:, j] /= T[:, j, j].unsqueeze(1)
            if j + 1 < c:
                T[:, j + 1:, j + 1:] -= T[:, j + 1:, j: j + 1] * T[:, j: j + 1, j + 1:]
    return T, order


def tournament(P, leaf, levels):
    """(selected rows in pivot order, their factored block) of panel P."""
    m, c = P.shape

    def play(rows):                       # equal-sized row sets, one batch
        T, order = gepp(P[rows])
        k = min(rows.shape[1], c)
        return rows.gather(1, order[:, :k]), T

    full, T = m // leaf, None
    sets = []
    if full:
        got, T = play(torch.arange(full * leaf, device=P.device).view(full, leaf))
        sets = list(got)
    if m % leaf:
        got, T = play(torch.arange(full * leaf, m, device=P.device).view(1, -1))
        sets += list(got)
    for groups in rounds(len(sets), levels):
        stacked = [torch.cat([sets[i] for i in g]) for g in groups]
        new = [s if len(g) == 1 else None for s, g in zip(stacked, groups)]
        sizes = {len(s) for s, n in zip(stacked, new) if n is None}
        for size in sizes:
            which = [i for i, s in enumerate(stacked) if new[i] is None and len(s) == size]
            got, T = play(torch.stack([stacked[i] for i in which]))
            for i, g in zip(which, got):
                new[i] = g
        sets = new
    return sets[0], T[0]


def exact_lu(A, b, leaf, levels):
    A = A.clone()
    m, n = A.shape
    K = min(m, n)
    ipiv = torch.zeros(K, dtype=torch.int32)
    for kb in range(0, K, b):
        bk = min(b, K - kb)
        sel, T = tournament(A[kb:, kb: kb + bk], leaf, levels)
        sel, at, where = sel.tolist(), {}, {}
        for i in range(bk):               # the swap sequence that brings row sel[i] to place i
            p = where.get(sel[i], sel[i])
            ipiv[kb + i] = kb + p + 1
            here = at.get(i, i)
            at[p], where[here] = here, p
            at[i], where[sel[i]] = sel[i], i
        dst = torch.tensor(sorted(at), device=A.device)
        src = torch.tensor([at[d] for d in sorted(at)], device=A.device)
        A[kb + dst] = A[kb + src]
        A[kb: kb + bk, kb: kb + bk] = T[:bk, :bk]
        U = T[:bk, :bk].triu()
        if kb + bk < m:
            A[kb + bk:, kb: kb + bk] = torch.linalg.solve_triangular(U, A[kb + bk:, kb: kb + bk], upper=True, left=False)
        if kb + bk < n:
            A[kb: kb + bk, kb + bk:] = torch.linalg.solve_triangular(T[:bk, :bk], A[kb: kb + bk, kb + bk:], upper=False,
                                                                      unitriangular=True)
            A[kb + bk:, kb + bk:] -= A[kb + bk:, kb: kb + bk] @ A[kb: kb + bk, kb + bk:]
    return A, ipiv


def house(T):
    """Householder QR of a batch: (V unit-lower, R, T of Q = I - V T V^T)."""
    T = T.clone()
    nb, r, c = T.shape
    k = min(r, c)
    V = torch.zeros(nb, r, k, dtype=T.dtype, device=T.device)
    tau = torch.zeros(nb, k, dtype=T.dtype, device=T.device)
    for j in range(k):
        x = T[:, j:, j]
        alpha, rest = x[:, 0], x[:, 1:].square().sum(1)
        beta = -torch.copysign((alpha.square() + rest).sqrt(), alpha)
        some = rest > 0
        tau[:, j] = torch.where(some, (beta - alpha) / beta, 0.0)
        v = x / torch.where(some, alpha - beta, 1.0).unsqueeze(1)
        v[:, 0] = 1.0
        v[~some, 1:] = 0.0
        V[:, j:, j] = v
        T[:, j:, j:] -= tau[:, j].view(-1, 1, 1) * v.unsqueeze(2) * torch.einsum("bi,bij->bj", v, T[:, j:, j:]).unsqueeze(1)
    W = torch.zeros(nb, k, k, dtype=T.dtype, device=T.device)
    Z = V.transpose(1, 2) @ V
    for j in range(k):
        W[:, :j, j] = -tau[:, j: j + 1] * torch.einsum("bij,bj->bi", W[:, :j, :j], Z[:, :j, j])
        W[:, j, j] = tau[:, j]
    return V, T[:, :k].triu(), W


def exact_qr(A, b, leaf, levels, B=None):
    """(A in caqr_factor's storage, qtree, Q^T B in place of B)."""
    A = A.clone()
    B = None if B is None else B.clone()
    m, n = A.shape
    qtree = []
    for kb in range(0, n, b):
        bk = min(b, n - kb)
        P = A[kb:, kb: kb + bk].clone()
        mk = m - kb
        rest = [C for C in (A[kb:, kb + bk:], None if B is None else B[kb:]) if C is not None and C.shape[1]]

        def node(rows):                    # rows: nodes x r indices; R sits in each child's top rows
            V, R, W = house(P[rows])
            for C in rest:
                X = C[rows]
                C[rows.reshape(-1)] = (X - V @ (W.transpose(1, 2) @ (V.transpose(1, 2) @ X))).reshape(-1, C.shape[1])
            blocks = torch.zeros(len(rows), b, b, dtype=A.dtype, device=A.device)
            blocks[:, :W.shape[1], :W.shape[1]] = W
            return V, R, list(blocks.transpose(1, 2))       # column-major blocks

        full = mk // leaf
        tops, Ts = [], []
        for lo, cnt, size in ((0, full, leaf), (full * leaf, 1 if mk % leaf else 0, mk % leaf)):
            if not cnt:
                continue
            rows = (lo + torch.arange(cnt * size, device=A.device)).view(cnt, size)
            V, R, T = node(rows)
            k = R.shape[1]
            F = V.clone() if k == bk else torch.cat([V, torch.zeros(cnt, size, bk - k, dtype=A.dtype, device=A.device)], 2)
            F = F.tril(-1)
            F[:, :k] += R
            P[rows.reshape(-1)] = F.reshape(-1, bk)
            A[kb + rows.reshape(-1), kb: kb + bk] = F.reshape(-1, bk)
            tops += list(rows[:, :k])
            Ts += T
        for groups in rounds(len(tops), levels):
            new = [tops[g[0]] if len(g) == 1 else None for g in groups]
            Tm = [None] * len(groups)
            sizes = {tuple(len(tops[i]) for i in g) for g in groups if len(g) > 1}
            for size in sizes:
                which = [i for i, g in enumerate(groups) if new[i] is None and tuple(len(tops[c]) for c in g) == size]
                rows = torch.stack([torch.cat([tops[c] for c in groups[i]]) for i in which])
                # below the diagonal of an R sit its node's reflectors: not part of the stack
                keep, offs = P[rows].clone(), [sum(size[:c]) for c in range(len(size) + 1)]
                for lo, hi in zip(offs, offs[1:]):
                    P[rows[:, lo:hi].reshape(-1)] = keep[:, lo:hi].triu().reshape(-1, bk)
                V, R, T = node(rows)
                k = R.shape[1]
                for c, (lo, hi) in enumerate(zip(offs, offs[1:])):
                    low = keep[:, lo:hi].tril(-1)
                    up = R[:, :hi] if c == 0 else V[:, lo:hi].triu()
                    F = low + up.triu()
                    P[rows[:, lo:hi].reshape(-1)] = F.reshape(-1, bk)
                    A[kb + rows[:, lo:hi].reshape(-1), kb: kb + bk] = F.reshape(-1, bk)
                for t, i in enumerate(which):
                    new[i], Tm[i] = rows[t, :k], T[t]
            tops = new
            Ts += [t for t in Tm if t is not None]
        qtree += Ts
    return A, torch.stack(qtree).reshape(-1), B


def exact(case, seed):
    kind = case["work"]
    if kind == "batch":
        return None                        # thousands of shapes, one by one: minutes
    m, n = shape(case)
    s = prepare(case, seed)
    A, B = s["A"].contiguous(), s.get("B")
    if kind == "gesv":                     # the factors are of reduced precision by choice
        return torch.linalg.solve(A, B), None, None, None
    if kind == "gels":
        Q, R = torch.linalg.qr(A)
        return torch.linalg.solve_triangular(R, Q.t() @ B, upper=True), None, None
    leaf, levels = parse_tree(case["tree"])
    b = min(case.get("b", n), n)
    leaf = max(leaf, case.get("b", 1))
    if kind in ("tsqr", "qr", "qr_solve"):
        F, qtree, QB = exact_qr(A, b, leaf, levels, B)
        if case.get("b", n) > n:           # T blocks of b x b with the panel's in the corner
            blocks = qtree.view(-1, b, b)
            qtree = torch.zeros(len(blocks), case["b"], case["b"], dtype=A.dtype, device=DEV)
            qtree[:, :b, :b] = blocks
            qtree = qtree.reshape(-1)
        if B is None:
            return F, qtree, None
        QB[:n] = torch.linalg.solve_triangular(F[:n].triu(), QB[:n], upper=True)
        return F, qtree, None, QB
    F, _ = exact_lu(A, b, leaf, levels)
    if B is None:
        return F, None, None
    return F, None, None, torch.linalg.solve(A, B)
