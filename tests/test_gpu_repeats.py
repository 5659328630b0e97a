"""A presolve repeats its result bit for bit, the sign of a zero included."""
import numpy as np
import pytest

from lpmake import INF
from paper_2609_16182_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402


def zero_ties(k, seed=0):
    """k columns x in [-5, 5], each in four rows that imply x >= 0 (x + s >= 0 and -x - s <= 0 with s a
    sum of columns in [-1, 0], as long as the row) and four that imply x <= 0: half of the implied
    bounds come out as -0.  The rows stand in a random order."""
    r = np.random.default_rng(seed)
    rows, lhs, rhs = [], [], []
    for j in range(k):
        for t in range(8):
            pad = k + r.choice(2 * k, int(r.choice([1, 1, 2, 6, 30])), replace=False)
            low = t < 4
            if low:  # pads in [-1, 0]: x >= -max(pads) = 0
                s, sides = (1.0, (0.0, INF)) if t % 2 else (-1.0, (-INF, 0.0))
                rows.append([(j, s)] + [(int(p), s) for p in pad])
            else:    # -pads in [0, 1]: x <= 0
                s, sides = (1.0, (-INF, 0.0)) if t % 2 else (-1.0, (0.0, INF))
                rows.append([(j, s)] + [(int(p), -s) for p in pad])
            lhs.append(sides[0])
            rhs.append(sides[1])
    order = r.permutation(len(rows))
    rows = [sorted(rows[i]) for i in order]
    n = 3 * k
    lb, ub = np.full(n, -1.0), np.zeros(n)
    lb[:k], ub[:k] = -5.0, 5.0
    lens = [len(x) for x in rows]
    return synth.LP(m=len(rows), n=n, row_ptr=np.concatenate([[0], np.cumsum(lens)]).astype(np.int32),
                    col_idx=np.array([j for x in rows for j, _ in x], np.int32),
                    val=np.array([a for x in rows for _, a in x]), c=np.ones(n), lhs=np.array(lhs)[order],
                    rhs=np.array(rhs)[order], lb=lb, ub=ub)


@pytest.mark.parametrize("kw", [{}, {"timing": 1}, {"dual_records": 1}, {"dual_fixing": 1}], ids=str)
def test_zero_bounds_repeat(kw):
    lp = zero_ties(2500)
    first = None
    for _ in range(12):
        g = lpp.presolve(lp, max_rounds=1, **kw)
        got = [np.ascontiguousarray(getattr(g, f)).tobytes() for f in ("col_lb", "col_ub", "col_val")]
        first = first or got
        assert got == first
    b = lpp.presolve_batch([lp, lp], max_rounds=1, **kw)
    for x in b:
        assert [np.ascontiguousarray(getattr(x, f)).tobytes() for f in ("col_lb", "col_ub", "col_val")] == first
