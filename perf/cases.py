"""The calls that performance is measured on.

Each case is one use of the library through its public entry points, on a
synthetic LP of the kinds the benchmark and the tests use (``synth.py``): the
small planted mix, the skewed LP (row lengths 1 + Zipf(2), column weights
Zipf(1.8)) and the LP-relaxation-like matrix with dense columns.  The inputs
are drawn on the GPU from the seed alone; matrix values and the point x0 that
the sides are built around lie on binary grids, so that A x0 is summed in
integers and comes out the same on every run.

A presolve is a fixpoint iteration whose every round decides by comparisons,
so a full call has no 64-bit value that plain array code could give;
``exact`` covers the row activities.
"""
from __future__ import annotations

import ctypes as C

import numpy as np
import torch

from paper_2609_16182_gb300 import lpp, synth

DEV = "cuda"
INF = float("inf")
VAL_GRID = 2.0 ** 16   # matrix values are multiples of 1 / VAL_GRID
LAM_GRID = 2.0 ** 8    # factors of scaled copies
X_GRID = 2.0 ** 12     # bounds and x0
DOT_GRID = VAL_GRID * LAM_GRID * X_GRID  # products a_ij x_j, copies included: 36 bits

# entries per row of each kind of LP, nominal (the actual count is random)
PER_ROW = {"mix": 6.0, "skewed": 10.0, "relax": 16.0}
COLS_PER_ROW = {"mix": 1.5, "skewed": 1.5, "relax": 2.0}


def listed():
    return [
        # the smallest call: one 200-row LP, as an interactive caller or a branch-and-bound node has it
        {"name": "mix_200", "call": "presolve", "lp": "mix", "m": 200, "opts": ""},
        # an ordinary LP on the device (0.2M nonzeros, the middle of the serving range)
        {"name": "skewed_20k", "call": "presolve", "lp": "skewed", "m": 20011, "opts": ""},
        # the benchmark LP: 2M rows, 3M columns, 20M nonzeros, a few rows with a large share of them
        {"name": "skewed_2m", "call": "presolve", "lp": "skewed", "m": 2000000, "opts": ""},
        # the LP-relaxation workload at its full size: dense columns, scaled row copies, many rounds
        {"name": "relax_500k", "call": "presolve", "lp": "relax", "m": 500000, "opts": ""},
        # doubleton equations substituted out (rows rewritten, A^T rebuilt)
        {"name": "relax_doubletons_250k", "call": "presolve", "lp": "relax", "m": 250007, "opts": "doubletons"},
        # parallel columns merged (1% scaled column copies)
        {"name": "skewed_parcols_500k", "call": "presolve", "lp": "skewed", "m": 500009, "opts": "parallel_cols"},
        # the dual explorers together: free column singletons and dual fixing by locks
        {"name": "skewed_dualexp_500k", "call": "presolve", "lp": "skewed", "m": 500009,
         "opts": "col_singletons,dual_fixing"},
        # host arrays in, reduced LP out to the host, a reduced solution mapped back (a CPU solver's use)
        {"name": "host_skewed_200k", "call": "roundtrip", "lp": "skewed", "m": 200003, "opts": ""},
        # the same with row duals and reduced costs (records of the rows behind tightened bounds)
        {"name": "host_dual_20k", "call": "roundtrip", "lp": "skewed", "m": 20011, "opts": "dual_records"},
        # the ragged batch: 4,096 LPs of 50 to 5,000 rows, the reduced LPs read on the device
        {"name": "batch_4096", "call": "batch", "lp": "mix", "m": 5000, "count": 4096, "opts": ""},
        # a burst of requests to the server, 1e3 to 1e5 nonzeros each
        {"name": "serve_32", "call": "serve", "lp": "skewed", "m": 10000, "count": 32, "opts": ""},
        # row activities alone, for a solver that allocates nothing (20M nonzeros)
        {"name": "activity_2m", "call": "activity", "lp": "skewed", "m": 2000000, "opts": ""},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    kind = rng.choice(["mix", "skewed", "skewed", "skewed", "relax", "opt", "roundtrip", "batch", "serve", "activity"])
    if kind == "mix":
        return {"call": "presolve", "lp": "mix", "m": size(50, 5000), "opts": ""}
    if kind == "skewed":
        return {"call": "presolve", "lp": "skewed", "m": size(100, 1900000), "opts": ""}
    if kind == "relax":
        return {"call": "presolve", "lp": "relax", "m": size(1000, 480000),
                "opts": rng.choice(["", "", "doubletons"])}
    if kind == "opt":
        return {"call": "presolve", "lp": "skewed", "m": size(1000, 480000),
                "opts": rng.choice(["parallel_cols", "col_singletons", "dual_fixing", "dual_records",
                                    "col_singletons,dual_fixing", "parallel_cols,col_singletons,dual_fixing"])}
    if kind == "roundtrip":
        dual = rng.random() < 0.5
        return {"call": "roundtrip", "lp": "skewed", "m": size(100, 19000 if dual else 190000),
                "opts": "dual_records" if dual else ""}
    if kind == "batch":
        return {"call": "batch", "lp": "mix", "m": size(100, 5000), "count": size(16, 4000), "opts": ""}
    if kind == "serve":
        return {"call": "serve", "lp": "skewed", "m": size(1000, 10000), "count": size(4, 32), "opts": ""}
    return {"call": "activity", "lp": "skewed", "m": size(100, 1900000), "opts": ""}


# ------------------------------------------------------------------ generators
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _rand(g, k):
    return torch.rand(int(k), generator=g, device=DEV, dtype=torch.float64)


def _randn(g, k):
    return torch.randn(int(k), generator=g, device=DEV, dtype=torch.float64)


def _grid(x, q):
    return torch.round(x * q) / q


def _ptr(lengths):
    p = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lengths, 0, out=p[1:])
    return p


def _perm(g, k):
    return torch.argsort(_rand(g, k), stable=True)


def _zipf(g, s, size, cap):
    """k in 1..cap with P(k) ~ k^-s, the tail on the cap."""
    zeta = {2.0: 1.6449340668482264, 1.8: 1.8822296181028220}[s]
    cdf = np.cumsum(np.arange(1, cap, dtype=np.float64) ** -s) / zeta
    return 1 + torch.searchsorted(torch.from_numpy(cdf).to(DEV), _rand(g, size), right=True)


def _lognormal(g, k):
    mag = _grid(torch.exp(_randn(g, k)), VAL_GRID).clamp_(min=1.0 / VAL_GRID)
    return torch.where(_rand(g, k) < 0.5, -mag, mag)


def _magnitudes(g, k, hi):
    v = _grid((2.0 * _rand(g, k) - 1.0) * hi, VAL_GRID)
    return torch.where(v.abs() < 1e-2, torch.full_like(v, 1e-2).mul_(VAL_GRID).ceil_().div_(VAL_GRID), v)


def _distinct(rows, cols, n, fixed, redraw):
    """Columns drawn again until every row holds distinct ones (entries
    marked fixed keep theirs); redraw(positions, pass) gives new columns."""
    for it in range(200):
        key, order = torch.sort(rows * n + cols, stable=True)
        dup = torch.nonzero(key[1:] == key[:-1]).flatten()
        if dup.numel() == 0:
            return cols
        a, b = order[dup], order[dup + 1]
        redo = torch.unique(torch.where(fixed[b], a, b)) if fixed is not None else b
        cols[redo] = redraw(redo, it)
    raise RuntimeError("column assignment did not converge")


def _sort_rows(rows, cols, vals, m, n):
    key, order = torch.sort(rows * n + cols)
    return _ptr(torch.bincount(rows, minlength=m)), key % n, vals[order], key // n


def _int_dot(rows, a, x, m):
    """sum a x per row, exactly: the products are multiples of 1 / DOT_GRID."""
    t = torch.round(a * x * DOT_GRID).to(torch.int64)
    s = torch.zeros(m, dtype=torch.int64, device=DEV)
    s.index_add_(0, rows, t)
    return s.to(torch.float64) / DOT_GRID


def _point(g, lb, ub):
    fl, fu = torch.isfinite(lb), torch.isfinite(ub)
    l0, u0 = torch.where(fl, lb, 0.0), torch.where(fu, ub, 0.0)
    both = l0 + _rand(g, lb.numel()) * (u0 - l0)
    x = torch.where(fl & fu, both, torch.where(fl, l0 + 1.0, torch.where(fu, u0 - 1.0, _randn(g, lb.numel()))))
    return _grid(x, X_GRID)


def _sides(g, ax, eq):
    """Around A x0: equalities, else a lognormal slack on each side, one of
    them dropped with probability 0.3."""
    m = ax.numel()
    lhs = ax - torch.exp(_randn(g, m)) * (1.0 + ax.abs())
    rhs = ax + torch.exp(_randn(g, m)) * (1.0 + ax.abs())
    drop, which = _rand(g, m) < 0.3, _rand(g, m) < 0.5
    lhs = torch.where(drop & which, -INF, lhs)
    rhs = torch.where(drop & ~which, INF, rhs)
    return torch.where(eq, ax, lhs), torch.where(eq, ax, rhs)


def _cost(g, lb, ub):
    """U[-1, 1], signed so that no variable can lower it without limit."""
    c = 2.0 * _rand(g, lb.numel()) - 1.0
    fl, fu = torch.isfinite(lb), torch.isfinite(ub)
    c = torch.where(fl & ~fu, c.abs(), torch.where(~fl & fu, -c.abs(), c))
    return torch.where(~fl & ~fu, 0.0, c)


def _lp(m, n, ptr, cols, vals, c, lhs, rhs, lb, ub):
    return synth.LP(m=m, n=n, row_ptr=ptr.to(torch.int32), col_idx=cols.to(torch.int32), val=vals.contiguous(),
                    c=c.contiguous(), lhs=lhs.contiguous(), rhs=rhs.contiguous(), lb=lb.contiguous(),
                    ub=ub.contiguous())


def skewed(seed, m, plant=()):
    """Row lengths 1 + Zipf(2) (capped, stretched to 10 m entries), 5% of
    them 1, column weights Zipf(1.8), every column at least one entry;
    lognormal values, 30% equalities, 20% infinite bounds, 3% rows planted
    redundant.  plant: 1% scaled column copies ("parallel_cols"), a free
    zero-cost singleton column in 30% of the equalities ("col_singletons")."""
    g = _gen(seed)
    n = max(15, int(1.5 * m))
    cap = max(2, min(500000, m // 4))
    ln = 1 + _zipf(g, 2.0, m, cap)
    total, target = int(ln.sum()), 10 * m
    if total < target:
        ln = torch.where(ln > 2, torch.round(ln * (target / total)).to(torch.int64).clamp_(max=cap), ln)
    ln = ln.clamp_(max=n)
    ln[_rand(g, m) < 0.05] = 1
    ptr = _ptr(ln)
    nnz = int(ptr[-1])
    rows = torch.repeat_interleave(torch.arange(m, device=DEV), ln)
    cum = torch.cumsum(_zipf(g, 1.8, n, max(2, m // 4)), 0)
    span = float(cum[-1])

    def by_weight(k):
        return torch.searchsorted(cum, (_rand(g, k) * span).to(torch.int64), right=True).clamp_(max=n - 1)

    cols = by_weight(nnz)
    fixed = torch.zeros(nnz, dtype=torch.bool, device=DEV)
    if nnz >= n:
        slots = _perm(g, nnz)[:n]
        cols[slots] = _perm(g, n)
        fixed[slots] = True
    cols = _distinct(rows, cols, n, fixed, lambda at, it: by_weight(at.numel()) if it < 3 else
                     (_rand(g, at.numel()) * n).to(torch.int64))
    vals = _lognormal(g, nnz)
    lb = _grid(-10.0 * _rand(g, n), X_GRID)
    ub = _grid(1.0 + 99.0 * _rand(g, n), X_GRID)
    lb[_rand(g, n) < 0.2] = -INF
    ub[_rand(g, n) < 0.2] = INF
    x0 = _point(g, lb, ub)
    c = _cost(g, lb, ub)
    ax = _int_dot(rows, vals, x0[cols], m)
    eq = _rand(g, m) < 0.3
    lhs, rhs = _sides(g, ax, eq)
    # redundant rows: one-sided, the side above sum |a_k b_k|
    need = torch.where(vals > 0, ub[cols], lb[cols])
    fin = torch.isfinite(need)
    crude = _int_dot(rows, vals.abs(), torch.where(fin, need.abs(), 0.0), m)
    bad = torch.zeros(m, dtype=torch.int64, device=DEV).index_add_(0, rows, (~fin).to(torch.int64))
    cand = torch.nonzero((bad == 0) & (ln >= 2)).flatten()
    red = cand[_perm(g, cand.numel())[:int(0.03 * m)]]
    rhs[red] = 1.0 + 2.0 * crude[red]
    lhs[red] = -INF
    if "parallel_cols" in plant:
        count = max(1, n // 100)
        lam_of = torch.zeros(n, dtype=torch.float64, device=DEV)
        base = _perm(g, n)[:count]
        lams = torch.tensor([-4.0, -2.0, -0.5, 0.5, 2.0, 4.0], dtype=torch.float64, device=DEV)
        lam_of[base] = lams[(_rand(g, count) * 6).to(torch.int64)]
        new = torch.full((n,), -1, dtype=torch.int64, device=DEV)
        new[base] = n + torch.arange(count, device=DEV)
        pick = torch.nonzero(lam_of[cols] != 0).flatten()
        rows = torch.cat([rows, rows[pick]])
        vals = torch.cat([vals, vals[pick] * lam_of[cols[pick]]])
        cols = torch.cat([cols, new[cols[pick]]])
        c = torch.cat([c, lam_of[base] * c[base]])
        lb = torch.cat([lb, torch.full((count,), -1.0, dtype=torch.float64, device=DEV)])
        ub = torch.cat([ub, torch.full((count,), 1.0, dtype=torch.float64, device=DEV)])
        n += count
    if "col_singletons" in plant:
        of = torch.nonzero(eq & torch.isfinite(lhs)).flatten()
        of = of[_perm(g, of.numel())[:int(0.3 * of.numel())]]
        k = of.numel()
        rows = torch.cat([rows, of])
        cols = torch.cat([cols, n + torch.arange(k, device=DEV)])
        vals = torch.cat([vals, _magnitudes(g, k, 5.0)])
        c = torch.cat([c, torch.zeros(k, dtype=torch.float64, device=DEV)])
        lb = torch.cat([lb, torch.full((k,), -INF, dtype=torch.float64, device=DEV)])
        ub = torch.cat([ub, torch.full((k,), INF, dtype=torch.float64, device=DEV)])
        n += k
    ptr, cols, vals, _ = _sort_rows(rows, cols, vals, m, n)
    return _lp(m, n, ptr, cols, vals, c, lhs, rhs, lb, ub)


def relax(seed, m):
    """LP-relaxation-like: 10 dense columns (200k entries at m = 500k), 5%
    scaled row copies, 4% doubleton equations, 2% loosened upper bounds,
    16 entries per row, n = 2 m."""
    g = _gen(seed)
    n = 2 * m
    dense, dense_len = 10, min(m, max(1, int(0.4 * m)))
    n_par = m // 20
    n_src = m - n_par
    order = _perm(g, n_src)
    is_dbl = torch.zeros(n_src, dtype=torch.bool, device=DEV)
    is_dbl[order[:m // 25]] = True
    src = order[m // 25:][_perm(g, n_src - m // 25)[:n_par]]  # the rows copied are no doubletons
    mean = torch.full((n_src,), (16.0 * m - dense * dense_len) / m - 2.0, device=DEV)
    ln = 2 + torch.poisson(mean, generator=g).to(torch.int64)
    ln[is_dbl] = 2
    ln = ln.clamp_(max=n - dense)
    rows = torch.repeat_interleave(torch.arange(n_src, device=DEV), ln)
    cols = dense + (_rand(g, rows.numel()) * (n - dense)).to(torch.int64)
    cols = _distinct(rows, cols, n, None,
                     lambda at, it: dense + (_rand(g, at.numel()) * (n - dense)).to(torch.int64))
    drows = torch.cat([_perm(g, n_src)[:dense_len] for _ in range(dense)])
    dcols = torch.repeat_interleave(torch.arange(dense, device=DEV), min(dense_len, n_src))
    keep = ~is_dbl[drows]
    rows, cols = torch.cat([rows, drows[keep]]), torch.cat([cols, dcols[keep]])
    ptr, cols, vals, rows = _sort_rows(rows, cols, _lognormal(g, rows.numel()), n_src, n)
    lam = _grid(0.5 + 3.5 * _rand(g, n_par), LAM_GRID)
    lam = torch.where(_rand(g, n_par) < 0.5, -lam, lam)
    ln = ptr[1:] - ptr[:-1]
    cl = ln[src]
    at = torch.repeat_interleave(ptr[src] - _ptr(cl)[:-1], cl) + torch.arange(int(cl.sum()), device=DEV)
    rows = torch.cat([rows, torch.repeat_interleave(torch.arange(n_src, m, device=DEV), cl)])
    cols = torch.cat([cols, cols[at]])
    vals = torch.cat([vals, vals[at] * torch.repeat_interleave(lam, cl)])
    place = _perm(g, m)
    eq0 = _rand(g, m) < 0.3
    eq0[:n_src] |= is_dbl
    eq0[n_src:] = eq0[src]
    eq = torch.empty_like(eq0)
    eq[place] = eq0
    ptr, cols, vals, rows = _sort_rows(place[rows], cols, vals, m, n)
    lb = torch.zeros(n, dtype=torch.float64, device=DEV)
    ub = _grid(1.0 + 99.0 * _rand(g, n), X_GRID)
    ub[_rand(g, n) < 0.1] = INF
    x0 = _point(g, lb, ub)
    lhs, rhs = _sides(g, _int_dot(rows, vals, x0[cols], m), eq)
    loose = (_rand(g, n) < 0.02) & (torch.arange(n, device=DEV) >= dense)
    ub = torch.where(loose, ub * 1024.0, ub)
    return _lp(m, n, ptr, cols, vals, _cost(g, lb, ub), lhs, rhs, lb, ub)


def mix(seed, ms, mean_len=6.0):
    """The planted mix, one LP per entry of ms (rows; n = 1.5 rows), drawn
    together: base rows of 2 .. 2 mean - 2 entries, and per 200 rows 10 empty,
    15 singleton and 10 redundant rows, 8 scaled copies, 20 fixed columns."""
    g = _gen(seed)
    k = len(ms)
    mk = torch.tensor(ms, dtype=torch.int64, device=DEV)
    nk = (mk * 3) // 2
    ro, co = _ptr(mk), _ptr(nk)
    M, N = int(ro[-1]), int(co[-1])
    lp_r = torch.repeat_interleave(torch.arange(k, device=DEV), mk)
    lp_c = torch.repeat_interleave(torch.arange(k, device=DEV), nk)

    def ranks(lp, off, cnt):  # a random order inside each LP: rank of each, and the member at each rank
        o = _perm(g, cnt)
        o = o[torch.argsort(lp[o], stable=True)]
        r = torch.empty_like(o)
        r[o] = torch.arange(cnt, device=DEV)
        return r - off[lp], o

    def per(x):
        return ((mk * x) // 200).clamp_(min=1)

    ends = torch.cumsum(torch.stack([per(10), per(15), per(10), per(8)]), 0)[:, lp_r]
    rank, at_rank = ranks(lp_r, ro, M)
    empty, single = rank < ends[0], (rank >= ends[0]) & (rank < ends[1])
    redundant, copy = (rank >= ends[1]) & (rank < ends[2]), (rank >= ends[2]) & (rank < ends[3])
    src = torch.arange(M, device=DEV)
    src[copy] = at_rank[(ro[lp_r] + ends[3] + rank - ends[2])[copy]]  # the base row as many ranks after the copies
    hi = max(3, int(round(2 * mean_len - 2)))
    ln = 2 + (_rand(g, M) * (hi - 1)).to(torch.int64)
    ln = torch.where(redundant, 2 + (_rand(g, M) * 4).to(torch.int64), ln)
    ln[single] = 1
    ln[empty | copy] = 0
    lb = torch.zeros(N, dtype=torch.float64, device=DEV)
    ub = _grid(1.0 + 99.0 * _rand(g, N), X_GRID)
    ub[_rand(g, N) < 0.1] = INF
    crank, _ = ranks(lp_c, co, N)
    fix = crank < per(20)[lp_c]
    fv = _grid(1.0 + 9.0 * _rand(g, N), X_GRID)
    lb, ub = torch.where(fix, fv, lb), torch.where(fix, fv, ub)
    finite = torch.nonzero(torch.isfinite(ub)).flatten()
    fo = _ptr(torch.bincount(lp_c[finite], minlength=k))
    rows = torch.repeat_interleave(torch.arange(M, device=DEV), ln)

    def columns(at, it=0):
        r = rows[at]
        lp = lp_r[r]
        u = _rand(g, at.numel())
        any_col = co[lp] + (u * nk[lp]).to(torch.int64)
        fin_col = finite[fo[lp] + (u * (fo[lp + 1] - fo[lp])).to(torch.int64)]
        return torch.where(redundant[r], fin_col, any_col)

    cols = _distinct(rows, columns(torch.arange(rows.numel(), device=DEV)), N, None, columns)
    vals = _magnitudes(g, rows.numel(), 10.0)
    p0 = _ptr(ln)
    lam = _grid(0.5 + 3.5 * _rand(g, M), LAM_GRID)
    lam = torch.where(_rand(g, M) < 0.5, -lam, lam)
    cr = torch.nonzero(copy).flatten()
    cl = ln[src[cr]]
    at = torch.repeat_interleave(p0[src[cr]] - _ptr(cl)[:-1], cl) + torch.arange(int(cl.sum()), device=DEV)
    rows = torch.cat([rows, torch.repeat_interleave(cr, cl)])
    cols = torch.cat([cols, cols[at]])
    vals = torch.cat([vals, vals[at] * torch.repeat_interleave(lam[cr], cl)])
    ptr, cols, vals, rows = _sort_rows(rows, cols, vals, M, N)
    x0 = _point(g, lb, ub)
    eq = _rand(g, M) < 0.5
    eq = eq[src]
    lhs, rhs = _sides(g, _int_dot(rows, vals, x0[cols], M), eq)
    big = _int_dot(rows, vals.abs(), torch.where(torch.isfinite(ub), ub, 0.0)[cols], M)
    margin = 1.0 + _rand(g, M) * big
    lhs = torch.where(redundant, torch.where(_rand(g, M) < 0.7, -big - margin, -INF), lhs)
    rhs = torch.where(redundant, big + margin, rhs)
    lhs = torch.where(empty, torch.where(_rand(g, M) < 0.7, -5.0 * _rand(g, M), -INF), lhs)
    rhs = torch.where(empty, torch.where(_rand(g, M) < 0.7, 5.0 * _rand(g, M), INF), rhs)
    c = _cost(g, lb, ub)
    # one set of arrays, cut into the LPs
    ent = ptr[ro]
    local = (ptr[:-1] - ent[lp_r]).to(torch.int32)
    cols = (cols - co[lp_r[rows]]).to(torch.int32)
    out = []
    hro, hco, hen = ro.tolist(), co.tolist(), ent.tolist()
    rps = torch.zeros(M + k, dtype=torch.int32, device=DEV)
    rps[torch.arange(M, device=DEV) + lp_r] = local
    rps[ro[1:] + torch.arange(k, device=DEV)] = (ent[1:] - ent[:-1]).to(torch.int32)
    for q in range(k):
        r, s = slice(hro[q], hro[q + 1]), slice(hco[q], hco[q + 1])
        z = slice(hen[q], hen[q + 1])
        out.append(synth.LP(m=hro[q + 1] - hro[q], n=hco[q + 1] - hco[q], row_ptr=rps[hro[q] + q:hro[q + 1] + q + 1],
                            col_idx=cols[z], val=vals[z], c=c[s], lhs=lhs[r], rhs=rhs[r], lb=lb[s], ub=ub[s]))
    return out


def _one(case, seed):
    m = case["m"]
    if case["lp"] == "mix":
        return mix(seed, [m], 9.0 if m <= 200 else 6.0)[0]
    if case["lp"] == "relax":
        return relax(seed, m)
    return skewed(seed, m, [w for w in ("parallel_cols", "col_singletons") if w in case["opts"]])


def _sizes(case):
    """Rows of each LP of a batch or a burst, log-uniform up to m."""
    lo = 50 if case["call"] == "batch" else 100
    r = np.random.default_rng(case["count"])
    return [int(x) for x in np.exp(r.uniform(np.log(lo), np.log(case["m"]), case["count"]))]


def _room(case):
    """Rows, columns and entries that hold any LP of the case."""
    if "count" in case:
        ms = _sizes(case)
        return sum(ms), sum(int(1.5 * m) for m in ms), sum(int(1.6 * PER_ROW[case["lp"]] * m) + 1000 for m in ms)
    m = case["m"]
    n = max(15, int(COLS_PER_ROW[case["lp"]] * m))
    if "parallel_cols" in case["opts"]:
        n += max(1, n // 100)
    if "col_singletons" in case["opts"]:
        n += m // 5
    return m, n, int(1.6 * PER_ROW[case["lp"]] * m) + 1000


# ----------------------------------------------------------------------- state
I32, F64 = torch.int32, torch.float64
CSR = {"row_ptr": I32, "col_idx": I32, "val": F64, "c": F64, "lhs": F64, "rhs": F64, "lb": F64, "ub": F64}
MAPS = {"row_map": I32, "col_map": I32}
CSC = {"csc_ptr": I32, "csc_idx": I32, "csc_val": F64}


def _buffers(case, fields, ptr_extra=1, **kw):
    """The solver's own arrays, into which the reduced LP is copied: as large
    as any LP of the case, zero past its end."""
    m, n, z = _room(case)
    size = {"row_ptr": m + ptr_extra, "col_idx": z, "val": z, "c": n, "lhs": m, "rhs": m, "lb": n, "ub": n,
            "row_map": m, "col_map": n, "csc_ptr": n + 1, "csc_idx": z, "csc_val": z}
    return {k: torch.zeros(size[k], dtype=t, **kw) for k, t in fields.items()}


def prepare(case, seed):
    flags = {w: 1 for w in case["opts"].split(",") if w}
    call = case["call"]
    state = {"call": call, "opts": lpp.opts(**flags)}
    if call == "presolve":
        state["lp"] = _one(case, seed)
        state["stream"] = torch.cuda.Stream()  # the caller's stream: the copies below follow the presolve on it
        state["opts"].stream = state["stream"].cuda_stream
        state["out"] = _buffers(case, {**CSR, **MAPS, **CSC}, device=DEV)
    elif call == "roundtrip":
        d = _one(case, seed)
        pinned = {k: v.cpu().pin_memory() for k, v in d.arrays().items()}
        state["pinned"] = pinned
        state["lp"] = synth.LP(m=d.m, n=d.n, **{k: v.numpy() for k, v in pinned.items()})
        state["out"] = _buffers(case, {**CSR, **MAPS}, device="cpu")
        # a reduced solution, as the solver after the presolve would have it
        r = lpp.presolve(state["lp"], state["opts"])
        red = r.reduced(csc=False)
        rng = np.random.default_rng(seed)
        state["x"] = np.clip(rng.normal(0.0, 10.0, red.n), red.lb, red.ub)
        state["y"] = rng.normal(0.0, 1.0, red.m)
        state["dual"] = bool(flags.get("dual_records"))
        r.close()
    elif call == "batch":
        state["lps"] = lpp.pack_lps(mix(seed, _sizes(case)))
        state["out"] = _buffers(case, CSR, case["count"], device=DEV)
    elif call == "serve":
        state["lps"] = [skewed(seed * 1009 + q, m) for q, m in enumerate(_sizes(case))]
        state["server"] = lpp.Server(4 << 30, state["opts"])
        state["out"] = _buffers(case, CSR, case["count"], device=DEV)
    else:
        d = _one(case, seed)
        state["lp"] = d
        state["out"] = {"act_min": torch.zeros(d.m, dtype=F64, device=DEV),
                        "act_max": torch.zeros(d.m, dtype=F64, device=DEV),
                        "ninf_min": torch.zeros(d.m, dtype=I32, device=DEV),
                        "ninf_max": torch.zeros(d.m, dtype=I32, device=DEV)}
        state["nnz"] = int(d.col_idx.numel())
    return state


class _Mem:
    """Device memory of the library as an array, for torch.as_tensor."""

    def __init__(self, ptr, count, dtype):
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": "<i4" if dtype is I32 else "<f8",
                                         "data": (ptr, False), "version": 3, "strides": None}


def _copy_reduced(res, out):
    """The reduced LP, its index maps and its A^T from the library's device
    memory into the caller's arrays."""
    L = lpp.load()
    v = res.device_view()
    rm, cm, tp, ti, tv = (C.c_void_p() for _ in range(5))
    if L.lpp_reduced_maps(res._red, C.byref(rm), C.byref(cm), 1) < 0 or \
            L.lpp_reduced_csc(res._red, C.byref(tp), C.byref(ti), C.byref(tv), 1) < 0:
        raise RuntimeError(lpp.last_error())
    m, n, z = v.m, v.n, v.nnz
    for name, ptr, count in (("row_ptr", v.row_ptr, m + 1), ("col_idx", v.col_idx, z), ("val", v.val, z),
                             ("c", v.c, n), ("lhs", v.lhs, m), ("rhs", v.rhs, m), ("lb", v.lb, n), ("ub", v.ub, n),
                             ("row_map", rm.value, m), ("col_map", cm.value, n), ("csc_ptr", tp.value, n + 1),
                             ("csc_idx", ti.value, z), ("csc_val", tv.value, z)):
        if count and ptr:
            out[name][:count].copy_(torch.as_tensor(_Mem(ptr, count, out[name].dtype), device=DEV))
    return v.obj_offset


_VIEW = np.dtype({"names": [f[0] for f in lpp.LpStruct._fields_[:12]],
                  "formats": ["<i4", "<i4", "<i8"] + ["<u8"] * 8 + ["<f8"],
                  "offsets": [getattr(lpp.LpStruct, f[0]).offset for f in lpp.LpStruct._fields_[:12]],
                  "itemsize": C.sizeof(lpp.LpStruct)})


def _concatenate(handles, out):
    """Many reduced LPs one after the other in the caller's arrays, gathered
    on the device from where each lies (a batched solver's input)."""
    L = lpp.load()
    views = (lpp.LpStruct * len(handles))()
    size = C.sizeof(lpp.LpStruct)
    at = C.addressof(views)
    fill = L.lpp_reduced_view
    for h in handles:
        if fill(h, C.cast(at, C.POINTER(lpp.LpStruct)), 1) < 0:
            raise RuntimeError(lpp.last_error())
        at += size
    v = np.frombuffer(views, dtype=_VIEW)
    for count, names in ((v["m"] + 1, ("row_ptr",)), (v["nnz"], ("col_idx", "val")), (v["m"], ("lhs", "rhs")),
                         (v["n"], ("c", "lb", "ub"))):
        count = count.astype(np.int64)
        have = count > 0
        if not have.any():
            continue
        total = int(count.sum())
        start = np.cumsum(count) - count
        item = [4 if out[k].dtype is I32 else 8 for k in names]
        base = [int(v[k][have].min()) for k in names]
        # per array: element (from the array's lowest address) of each LP's first entry, less its place in the output
        first = torch.from_numpy(np.stack([(v[k].astype(np.int64) - b) // w - start
                                           for k, b, w in zip(names, base, item)])).to(DEV)
        lp = torch.repeat_interleave(torch.from_numpy(count).to(DEV), output_size=total)
        lane = torch.arange(total, device=DEV)
        for q, k in enumerate(names):
            span = int(((v[k][have].astype(np.int64) - base[q]) // item[q] + count[have]).max())
            torch.index_select(torch.as_tensor(_Mem(base[q], span, out[k].dtype), device=DEV), 0, lane + first[q][lp],
                               out=out[k][:total])
    torch.cuda.current_stream().synchronize()  # the results are freed next
    return {"m": v["m"].copy(), "n": v["n"].copy(), "nnz": v["nnz"].copy(), "offset": v["obj_offset"].copy()}


def run(state):
    call, out = state["call"], state["out"]
    if call == "presolve":
        res = lpp.presolve(state["lp"], state["opts"])
        i = res.info
        with torch.cuda.stream(state["stream"]):
            offset = _copy_reduced(res, out)
        res.close()
        return {**out, "offset": offset, "verdict": (i.status, i.rounds, i.m_red, i.n_red, i.nnz_red, i.s5_left)}
    if call == "roundtrip":
        res = lpp.presolve(state["lp"], state["opts"])
        red = res.reduced(copy=False, csc=False)
        for k, t in out.items():
            a = torch.from_numpy(getattr(red, k))
            t[:a.numel()].copy_(a)
        got = {**out, "offset": red.obj_offset}
        if state["dual"]:
            got["x"], got["y"], got["z"] = res.postsolve_dual(state["lp"], state["x"], state["y"])
        else:
            got["x"] = res.postsolve_primal(state["x"])
        res.close()
        return got
    L = lpp.load()
    if call == "batch":  # through the C ABI, as a native caller with 4,096 handles
        k = state["lps"].count
        reds, recs, per = (C.c_void_p * k)(), (C.c_void_p * k)(), (C.c_int32 * k)()
        if L.lpp_presolve_batch(state["lps"].arr, k, C.byref(state["opts"]), reds, recs, per) < 0:
            raise RuntimeError(lpp.last_error())
        got = {**out, **_concatenate(reds, out), "status": np.array(per)}
        L.lpp_free_results(reds, recs, k)
        return got
    if call == "serve":
        srv = state["server"]
        res = [srv.take(t) for t in [srv.submit(lp) for lp in state["lps"]]]
        got = {**out, **_concatenate([r._red for r in res], out)}
        for r in res:
            r.close()
        return got
    lp = state["lp"]
    st = L.lpp_row_activity_noalloc(lp.m, lp.n, state["nnz"], lp.row_ptr.data_ptr(), lp.col_idx.data_ptr(),
                                    lp.val.data_ptr(), lp.lb.data_ptr(), lp.ub.data_ptr(), 1e20,
                                    out["act_min"].data_ptr(), out["act_max"].data_ptr(), out["ninf_min"].data_ptr(),
                                    out["ninf_max"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    if st < 0:
        raise RuntimeError(lpp.last_error())
    return out


def work(case):
    """The input LP read once and the reduced LP (nominally four fifths of
    it) written once; two fused multiply-adds per entry."""
    rows = case["m"]
    if "count" in case:  # log-uniform sizes: their mean
        lo = 50 if case["call"] == "batch" else 100
        rows = float(case["count"] * (case["m"] - lo) / np.log(case["m"] / lo))
    nnz = PER_ROW[case["lp"]] * rows
    cols = COLS_PER_ROW[case["lp"]] * rows
    if case["call"] == "activity":
        return {"bytes": 12.0 * nnz + (4 + 24) * rows + 16.0 * cols, "flops": 4.0 * nnz}
    lp = 12.0 * nnz + 20.0 * rows + 24.0 * cols
    csc = 12.0 * nnz + 4.0 * cols if case["call"] == "presolve" else 0.0
    maps = 4.0 * rows + 4.0 * cols
    return {"bytes": lp + 0.8 * (lp + csc + maps), "flops": 4.0 * nnz}


def exact(case, seed):
    if case["call"] != "activity":
        return None
    d = _one(case, seed)
    a = {k: v.cpu().numpy() for k, v in d.arrays().items()}
    rows = np.repeat(np.arange(d.m), np.diff(a["row_ptr"]))
    l, u = a["lb"][a["col_idx"]], a["ub"][a["col_idx"]]
    pos = a["val"] > 0
    out = []
    for b in (np.where(pos, l, u), np.where(pos, u, l)):
        fin = np.isfinite(b)
        # values and bounds are on the grids: the sum is exact in integers
        t = np.rint(a["val"] * np.where(fin, b, 0.0) * (VAL_GRID * X_GRID)).astype(np.int64)
        s = np.concatenate([[0], np.cumsum(t)])
        out.append(((s[a["row_ptr"][1:]] - s[a["row_ptr"][:-1]]).astype(np.float64) / (VAL_GRID * X_GRID),
                    np.bincount(rows[~fin], minlength=d.m).astype(np.int32)))
    return {"act_min": out[0][0], "act_max": out[1][0], "ninf_min": out[0][1], "ninf_max": out[1][1]}
