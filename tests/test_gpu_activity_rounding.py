"""Row activities of 17 to 64 entries: no longer chains of additions than 8 and
16 lanes per row have.

A sum whose longest path has k roundings is off by at most about k units of 2^-53
of the sum of its terms' magnitudes; 17 to 32 entries in 8 chains of 4 and a
butterfly have 7, 33 to 64 in 16 chains 8.  The first term of each row is 1 and the
others lie just above half a unit of it, so that every addition of one to a sum
beyond 1 is off by half a unit: one chain of 16 is 15 of them off.
"""
from fractions import Fraction

import numpy as np
import pytest

from lpmake import INF, make

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402

LENS = [17, 18, 24, 25, 31, 32, 33, 34, 47, 48, 49, 63, 64]
TINY = 2.0 ** -53 * (1 + 2.0 ** -10)


def rows_lp():
    rows, at = [], 0
    for k in LENS:
        for big in {0, 1, k // 2, k - 1}:
            rows.append({at + t: (1.0 if t == big else TINY) for t in range(k)})
        at += k
    m = len(rows)
    return make(rows, [-INF] * m, [1.5] * m, [1.0] * at, [2.0] * at), rows


@pytest.mark.parametrize("how", ["one kernel", "launched", "batch"])
def test_roundings_of_an_activity(how):
    lp, rows = rows_lp()
    if how == "batch":
        r = lpp.presolve_batch([lp, lp], max_rounds=1)[1]
    else:
        r = lpp.presolve(lp, max_rounds=1, timing=int(how == "launched"))
    for i, row in enumerate(rows):
        units = (7 if len(row) <= 32 else 8) * Fraction(1, 2 ** 53)
        exact = sum(Fraction(a) for a in row.values())
        for got, want in ((r.act_min[i], exact), (r.act_max[i], 2 * exact)):
            assert abs(Fraction(float(got)) - want) <= units * want, (i, len(row))
