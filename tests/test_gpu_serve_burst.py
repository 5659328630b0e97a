"""Submissions to the server go on while a request is presolved: a burst is queued, and
can be batched, instead of trickling in behind each request."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402
from test_gpu_batch import to_device  # noqa: E402


def test_submissions_do_not_wait_for_the_request_being_presolved():
    lps = [to_device(synth.skewed_like(100 + k, 600000)) for k in range(4)]
    want = [lpp.presolve(lp) for lp in lps]
    alone, submit = [], []
    for _ in range(8):
        t = time.perf_counter()
        lpp.presolve(lps[0]).close()
        alone.append(time.perf_counter() - t)
    with lpp.Server(16 << 30) as srv:
        srv.take(srv.submit(lps[0])).close()
        tickets = []
        for k in range(48):
            t = time.perf_counter()
            tickets.append(srv.submit(lps[k % 4]))
            submit.append(time.perf_counter() - t)
        for k, t in enumerate(tickets):
            r, w = srv.take(t), want[k % 4]
            assert (r.status, r.rounds) == (w.status, w.rounds)
            np.testing.assert_array_equal(r.col_kind, w.col_kind)
            r.close()
    # behind a grid that holds every register, the copies of every third submission take a whole presolve
    assert np.percentile(submit, 75) < 0.5 * np.median(alone), (sorted(submit), np.median(alone))
