"""A batch of one LP is an arena like any other: it gets the LP's solo result
with host and device inputs, in the persistent kernel and per round."""
import pytest

from lpmake import INF, make

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402
from test_gpu_batch import same_result, to_device  # noqa: E402

LPS = {"mix": lambda: synth.mix(1),
       "long rows": lambda: synth.skewed(4, m=8000, n=12000, target_nnz=90_000, row_cap=9000),
       "no rows": lambda: make([], [], [], [-1, 0], [1, 2], [1.0, -1.0]),
       "infeasible": lambda: make([{0: 1.0, 1: 1.0}], [5], [INF], [0, 0], [1, 1])}


@pytest.mark.parametrize("kw", [{}, {"batch_persistent": 0}, {"dual_records": 1}, {"max_rounds": 1}, {"max_rounds": 0},
                                {"timing": 1}, {"parallel_cols": 1}, {"col_singletons": 1, "dual_fixing": 1},
                                {"doubletons": 1}], ids=str)
@pytest.mark.parametrize("name", LPS)
def test_batch_of_one(name, kw):
    lp = LPS[name]()
    want = lpp.presolve(lp, **{k: v for k, v in kw.items() if k != "batch_persistent"})
    for inp in (lp, to_device(lp)):
        res = lpp.presolve_batch([inp], **kw)
        assert len(res) == 1
        same_result(res[0], want)
        assert (res[0].status, res[0].where, res[0].index) == (want.status, want.where, want.index)
