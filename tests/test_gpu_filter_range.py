"""The single-precision filter of the implied bounds at the ends of single
precision's range, with opts.huge beyond it: a bound of (double)FLT_MAX, as
callers write for "no bound", must be tightened as any other, in every kernel."""
import numpy as np
import pytest

import oracle
from lpmake import INF, make
from parity import compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402

FLT_MAX = float(np.finfo(np.float32).max)
HI20 = 2.0 ** 128 * (1 - 2.0 ** -20)  # the upper 20 mantissa bits one, but the last
ENDS = [FLT_MAX, HI20, float(np.nextafter(2.0 ** 128, 0)), 2.0 ** 128, float(np.nextafter(HI20, 0)), 2.0 ** 127]


@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("v", ENDS)
def test_bounds_at_the_end_of_single_precision(v, timing):
    n = 400
    for k in (2, 20, 40, 100, 300):  # entries per row: 1, 2, 4 and 32 lanes, a block
        rows, lhs, rhs = [], [], []
        lb, ub = np.zeros(n), np.full(n, 5.0)
        ub[0], lb[1] = v, -v
        rest = {j: 1.0 for j in range(2, 1 + k)}
        rows += [{0: 1.0, **rest}, {1: 1.0, **rest}, {0: -2.0, **rest}, {1: -0.5, **rest}]
        lhs += [-INF, -10.0, -24.0, -INF]
        rhs += [10.0 + k, INF, INF, 12.0 + k]
        lp = make(rows, lhs, rhs, lb, ub, c=np.ones(n))
        o = oracle.presolve(lp, oracle.default_opts(huge=1e300, max_rounds=1))
        g = lpp.presolve(lp, huge=1e300, max_rounds=1, timing=timing)
        compare(g, o, lp)
        assert g.col_ub[0] < 1e10 and g.col_lb[1] > -1e10


@pytest.mark.parametrize("v", ENDS)
def test_batch_members_with_such_bounds(v):
    lps = [make([{0: 1.0, 1: 1.0}, {0: 1.0, 1: -1.0}], [-INF, -3.0], [10.0, INF], [0.0, 0.0], [v, 5.0], c=[1.0, 1.0])
           for _ in range(3)]
    for lp, g in zip(lps, lpp.presolve_batch(lps, huge=1e300)):
        compare(g, oracle.presolve(lp, oracle.default_opts(huge=1e300)), lp)
