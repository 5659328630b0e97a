"""One kernel for all rounds, the same rounds launched, the persistent batch and
the per-round batch: an LP gets the same bits from each (the objective constant,
whose terms a batch adds in another order, to the last digits)."""
import numpy as np
import pytest

from parity import _close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402
from test_gpu_kernel_edges import EDGES, build  # noqa: E402

LPS = {"edges": lambda: build(1, EDGES, 8200), "edges, many": lambda: build(2, EDGES * 7, 8200),
       "no long row": lambda: build(3, EDGES[:-3] * 4, 8200), "dense": lambda: build(4, [300] * 40, 300),
       "short rows": lambda: build(5, list(np.random.default_rng(5).integers(0, 70, 3000)), 2500),
       "skewed": lambda: synth.skewed(8, m=9000, n=13500, target_nnz=90000, row_cap=5000),
       "relaxation": lambda: synth.lprelax(2, m=6000, n=12000, target_nnz=96000, n_dense=2, dense_len=2500),
       "mix": lambda: synth.mix(9, m=3000, n=4000)}
REDUCED = ("row_ptr", "col_idx", "val", "c", "lhs", "rhs", "lb", "ub", "row_map", "col_map", "csc_ptr", "csc_idx", "csc_val")
RECORDS = ("row_kind", "row_round", "row_aux", "row_val", "col_kind", "col_round", "col_val", "col_lb", "col_ub", "act_min",
           "act_max", "ninf_min", "ninf_max")


@pytest.mark.parametrize("kw", [{}, {"dual_records": 1}, {"max_rounds": 2}, {"dual_reductions": 0}], ids=str)
@pytest.mark.parametrize("name", LPS)
def test_forms_agree_bit_for_bit(name, kw):
    lp = LPS[name]()
    one, launched = lpp.presolve(lp, **kw), lpp.presolve(lp, timing=1, **kw)
    forms = [launched, lpp.presolve_batch([lp, lp], batch_persistent=0, **kw)[1]]
    if not kw.get("dual_records"):
        forms.append(lpp.presolve_batch([lp, lp], **kw)[1])
    a = one.reduced()
    assert a.obj_offset == launched.reduced().obj_offset
    for form in forms:
        assert (one.status, one.rounds) == (form.status, form.rounds)
        b = form.reduced()
        for f in REDUCED:
            np.testing.assert_array_equal(getattr(a, f), getattr(b, f), err_msg=f)
        for f in RECORDS:
            np.testing.assert_array_equal(getattr(one, f), getattr(form, f), err_msg=f)
        _close([a.obj_offset], [b.obj_offset], what="offset")
    for f in ("round_nnz", "round_rows_removed", "round_cols_fixed", "round_bounds_changed"):
        np.testing.assert_array_equal(getattr(one, f), getattr(launched, f), err_msg=f)
    if kw.get("dual_records"):
        for f, v in one.bound_sources().items():
            np.testing.assert_array_equal(v, launched.bound_sources()[f], err_msg=f)
