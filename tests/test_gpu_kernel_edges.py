"""The kernels at the sizes where their splits change, against the oracle.

Rows at both ends of every length class (lanes, warp, block, chunks), column
counts and entry counts at the ends of sort tiles and digits, schedules at the
ends of their tiles, key groups that need later passes of every kind (grid,
halves of the table, one block), batches whose members leave classes empty,
primal postsolve on the device.  Coefficients are powers of two and bounds small
whole numbers, so every sum is exact in any order and the oracle's results have
to come out within the parity bar, its decisions exactly.
"""
import numpy as np
import pytest

import oracle
from lpmake import INF, make
from parity import compare
from paper_2609_16182_gb300 import synth
from test_zz_no_alloc import Dev, check_oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402

EDGES = [0, 1, 2, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 4096, 4097, 8193]


def build(seed, lens, n, exps=(-1, 0, 1, 2)):
    """Rows of these lengths over n columns; a whole point inside the bounds
    satisfies every row, a third of them with no slack to spare."""
    r = np.random.default_rng(seed)
    m = len(lens)
    ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    cols = np.concatenate([np.sort(r.choice(n, k, replace=False)) for k in lens] + [np.zeros(0, int)])
    vals = r.choice([-1.0, 1.0], cols.size) * 2.0 ** r.choice(exps, cols.size)
    lb = r.integers(-8, 1, n).astype(float)
    ub = lb + r.integers(0, 9, n)
    x = np.clip(np.round((lb + ub) / 2), lb, ub)
    lb[r.random(n) < 0.05] = -INF
    ub[r.random(n) < 0.05] = INF
    ax = np.zeros(m)
    np.add.at(ax, np.repeat(np.arange(m), lens), vals * x[cols])
    slack = r.choice([0.0, 1.0, 16.0, 4096.0], m)
    lhs, rhs = ax - slack, ax + r.permutation(slack)
    drop = r.random(m)
    lhs[drop < 0.4] = -INF
    rhs[drop > 0.7] = INF
    return synth.LP(m=m, n=n, row_ptr=ptr, col_idx=cols.astype(np.int32), val=vals,
                    c=r.integers(-3, 4, n).astype(float), lhs=lhs, rhs=rhs, lb=lb, ub=ub)


def check(lp, **kw):
    o = oracle.presolve(lp, oracle.default_opts(**{k: v for k, v in kw.items() if k != "timing"}))
    g = lpp.presolve(lp, **kw)
    compare(g, o, lp)
    return g


# timing=1 launches the rounds, without it an LP of these sizes goes into one kernel
@pytest.mark.parametrize("kw", [{}, {"timing": 1}, {"dual_records": 1}, {"dual_records": 1, "timing": 1},
                                {"dual_fixing": 1}, {"col_singletons": 1}, {"parallel_cols": 1}])
@pytest.mark.parametrize("lens", [EDGES, EDGES * 3, [17] * 255 + [65] * 33, [], [0], [1], [4097]])
def test_row_classes(lens, kw):
    check(build(len(lens), lens, 8200), **kw)


@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 511, 513, 65536, 65537])
@pytest.mark.parametrize("nnz", [511, 513, 2047, 2048, 2049, 7000])
def test_column_counts_and_entry_tiles(n, nnz, timing):
    k = min(n, 3)
    lens = [k] * (nnz // k) + ([nnz % k] if nnz % k else [])
    lp = build(n + nnz, lens, n)
    if n > 3:  # the last column has an entry
        lp.col_idx[lp.row_ptr[1] - 1] = n - 1
    check(lp, timing=timing)


@pytest.mark.parametrize("m", [2047, 2048, 2049, 4097])
def test_schedule_tiles(m):
    lens = np.random.default_rng(m).choice([0, 1, 3, 7, 20, 40, 70, 300], m, p=[.05, .1, .4, .3, .1, .03, .015, .005])
    check(build(m, list(lens), 3 * m), timing=1)


@pytest.mark.parametrize("seed", range(4))
def test_magnitudes(seed):
    """Coefficients from 2^-20 to 2^20 in one row: the filter in single
    precision rejects, keeps and leaves undecided."""
    lp = build(seed, list(np.random.default_rng(seed).integers(2, 33, 800)), 1500, exps=tuple(range(-20, 21)))
    a, b = check(lp), check(lp, timing=1)
    np.testing.assert_array_equal(a.col_lb, b.col_lb)
    np.testing.assert_array_equal(a.col_ub, b.col_ub)


# sizes of the key groups: rows over the same two columns, no two parallel
@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("groups", [[513], [700], [5000], [2] * 3000 + [9] * 200, [2] * 6000, [3] * 256 + [2] * 257])
def test_later_passes_on_parallel_rows(groups, timing):
    rows = []
    for g, size in enumerate(groups):
        rows += [{2 * g: 1.0, 2 * g + 1: float(k + 2)} for k in range(size)]
        rows += [{2 * g: 2.0, 2 * g + 1: 2.0 * (size + 1)}, {2 * g: -1.0, 2 * g + 1: -2.0}]
    n, m = 2 * len(groups), len(rows)
    check(make(rows, [-INF] * m, [float(10 + k % 7) for k in range(m)], [-INF] * n, [INF] * n), timing=timing)


def test_batch_members_with_empty_classes():
    lps = [build(1, EDGES[:-2], 8200), build(2, [4096] * 3, 5000), build(3, [1] * 33, 40), build(4, [5] * 513, 600),
           build(5, [2, 2048, 2, 33], 3000), build(6, [], 7), build(7, [0] * 5, 3)]
    for lp, r in zip(lps, lpp.presolve_batch(lps)):
        compare(r, oracle.presolve(lp), lp)


def test_per_round_batch_of_many_members():
    lps = [build(s, [2, 3, 1, 0, 4], 6) for s in range(900)]  # their counters are longer than one fetch takes
    res = lpp.presolve_batch(lps, batch_persistent=0)
    for k in range(0, 900, 53):
        compare(res[k], oracle.presolve(lps[k]), lps[k], arena_stats=True)


@pytest.mark.parametrize("n", [1, 255, 257, 8200])
def test_primal_postsolve_on_the_device(n):
    lp = build(n, [min(n, k) for k in EDGES], n)
    r = lpp.presolve(lp)
    red = r.reduced()
    x = np.random.default_rng(n).standard_normal(red.n)
    want = np.where(r.col_kind != 0, r.col_val, 0.0)
    want[red.col_map] = x
    np.testing.assert_array_equal(r.postsolve_primal(x), want)


@pytest.mark.parametrize("lens", [EDGES, EDGES[::-1] * 2, [512] * 9 + [513] * 9, [1] * 257])
def test_row_activities(lens):
    lp = build(9, lens, 8200)
    check_oracle(lp, Dev(lp).call(lpp.load()))
