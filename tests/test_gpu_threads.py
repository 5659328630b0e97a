"""Presolves from several host threads: each gets its result, and they overlap."""
import threading
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402
from test_gpu_batch import to_device  # noqa: E402


def run(threads, work):
    errors = []

    def guarded(k):
        try:
            work(k)
        except BaseException as e:  # noqa: BLE001  the main thread raises it
            errors.append(e)

    ts = [threading.Thread(target=guarded, args=(k,)) for k in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def test_threads_get_their_results():
    lps = [synth.mix(1), synth.skewed(1, m=20000, n=30000, target_nnz=200000, row_cap=9000),
           synth.skewed(3, m=3000, n=4500, target_nnz=30000, row_cap=2000), synth.mix(2, m=2000, n=3000)]
    dev = [to_device(lp) for lp in lps]
    want = [lpp.presolve(lp) for lp in dev]
    red = [w.reduced() for w in want]

    def work(k):
        for it in range(8):
            q = (k + it) % len(dev)
            r = lpp.presolve(dev[q], timing=int(it == 7))
            a, b = r.reduced(), red[q]
            for f in ("row_ptr", "col_idx", "val", "c", "lhs", "rhs", "lb", "ub", "obj_offset", "row_map", "col_map",
                      "csc_ptr", "csc_idx", "csc_val"):
                np.testing.assert_array_equal(getattr(a, f), getattr(b, f), err_msg=f)
            r.close()

    run(8, work)


def test_presolves_of_eight_threads_overlap():
    """Eight callers of an LP of 0.18 M entries, whose rounds are one kernel: no more than 0.6 of
    one caller's time per call (one after the other: 0.8, the host's part alone overlaps)."""
    lp = to_device(synth.skewed(1, m=20000, n=30000, target_nnz=200000, row_cap=9000))

    def per_call(threads, reps=24):
        def work(_):
            for _ in range(reps):
                lpp.presolve(lp).close()

        best = 1e9
        for _ in range(3):
            t = time.perf_counter()
            run(threads, work)
            best = min(best, (time.perf_counter() - t) / (threads * reps))
        return best

    per_call(8, 4)
    one, eight = per_call(1), per_call(8)
    assert eight < 0.6 * one, (one, eight)
