"""S5's later passes go on in one block while the others of the presolve's kernel
wait: hundreds of passes over long rows are progress, not a barrier that fails."""
import numpy as np
import pytest

from lpmake import INF
from paper_2609_16182_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402


@pytest.mark.parametrize("passes", [40, 600])
def test_many_passes_over_dense_rows_of_one_key(passes):
    """512 rows over the same 5,000 columns, all positive: one key.  They agree in all entries
    but the last, so each is compared to its end; every tenth is a multiple of its predecessor."""
    m, n = 512, 5000
    a = np.ones((m, n))
    a[:, -1] = 1.0 + np.arange(m) / 1024
    a[9::10] = 2.0 * a[8::10][:len(a[9::10])]
    lp = synth.LP(m=m, n=n, row_ptr=np.arange(0, m * n + 1, n, dtype=np.int32),
                  col_idx=np.tile(np.arange(n, dtype=np.int32), m), val=a.ravel(), c=np.ones(n),
                  lhs=np.full(m, -INF), rhs=4.0 * n + np.arange(m), lb=np.zeros(n), ub=np.full(n, 10.0))
    g = lpp.presolve(lp, par_max_iter=passes, max_rounds=1)
    w = lpp.presolve(lp, par_max_iter=passes, max_rounds=1, timing=1)
    assert g.s5_left == w.s5_left and (passes < m) == (g.s5_left > 0)
    assert (g.row_kind == lpp.ROW_PARALLEL).sum() > 0
    for k in ("row_kind", "row_aux", "row_val", "col_kind", "col_lb", "col_ub"):
        np.testing.assert_array_equal(getattr(g, k), getattr(w, k))
