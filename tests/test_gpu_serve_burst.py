"""A burst that outlasts the server's first requests is batched: submissions do not
wait for the request being presolved."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp, synth  # noqa: E402
from test_gpu_batch import to_device  # noqa: E402


def test_a_long_burst_of_middle_sized_requests_is_batched():
    lps = [to_device(synth.skewed_like(100 + k, 600000)) for k in range(4)]
    want = [lpp.presolve(lp) for lp in lps]
    with lpp.Server(16 << 30) as srv:
        srv.take(srv.submit(lps[0])).close()
        tickets = [srv.submit(lps[k % 4]) for k in range(80)]
        for k, t in enumerate(tickets):
            r, w = srv.take(t), want[k % 4]
            assert (r.status, r.rounds) == (w.status, w.rounds)
            np.testing.assert_array_equal(r.col_kind, w.col_kind)
            r.close()
        assert srv.stats()["ticks"] > 0 and srv.stats()["solo"] < 40
