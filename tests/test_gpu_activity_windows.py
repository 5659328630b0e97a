"""lpp_row_activity_noalloc: rows of 33 to 4096 entries belong to the window of
the entry array in which they start, wherever they stand."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_16182_gb300 import lpp  # noqa: E402
from test_gpu_kernel_edges import build  # noqa: E402
from test_zz_no_alloc import Dev, check_oracle  # noqa: E402

SHAPES = {
    "32, 33": [32] * 70 + [33] * 260 + [32, 33] * 20,
    "64, 65": [64] * 70 + [65] * 130,
    "128, 129": [128] * 33 + [129] * 65,
    "512, 513": [512] * 17 + [513] * 17 + [512, 513] * 8,
    "4096, 4097": [4096] * 3 + [4097] * 2 + [4096, 4097, 4096],
    "off by one": [1] + [4096] * 4 + [3, 4095, 65, 4097],
    "together among short rows": [1, 2, 3] * 300 + [300] * 256 + [2] * 500 + [2000] * 40 + [1] * 100,
    "many empty rows in a window": [65] * 20 + [0] * 2049 + [65] * 10 + [0] * 5000 + [4000, 130, 4097] + [0] * 3000 + [65],
    "the last row, over the window's end": [0] * 2500 + [4040] + [0] * 2500 + [100] + [0] * 9 + [66],
    "one row": [33],
    "no entry but in the last row": [0] * 3000 + [40],
    "many empty rows, short ones": [33] * 40 + [0] * 2049 + [34] * 50 + [0] * 3000 + [32, 33, 31] * 40,
}


@pytest.mark.parametrize("name", SHAPES)
def test_rows_in_windows(name):
    lp = build(len(name), SHAPES[name], 8200)
    d = Dev(lp)
    d.amin.fill_(np.nan)
    d.nmax.fill_(-7)
    check_oracle(lp, d.call(lpp.load()))


def test_time_follows_the_entries_not_the_rows_standing_together():
    """12 M entries: in rows of 513 to 4096 entries no more than four times as
    long as in rows of 4097, which are split by windows."""
    L = lpp.load()
    nnz, n = 12 * 2 ** 20, 1_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    ci = torch.randint(0, n, (nnz,), generator=g, device="cuda", dtype=torch.int32)
    v = torch.randn(nnz, generator=g, device="cuda", dtype=torch.float64)
    lb, ub = -torch.ones(n, device="cuda", dtype=torch.float64), torch.ones(n, device="cuda", dtype=torch.float64)
    ms = {}
    for k in (513, 1000, 4096, 4097):
        m = nnz // k
        ptr = torch.arange(0, (m + 1) * k, k, device="cuda", dtype=torch.int32)
        d, c = torch.empty(2 * m, device="cuda", dtype=torch.float64), torch.empty(2 * m, device="cuda", dtype=torch.int32)
        t = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            assert L.lpp_row_activity_noalloc(m, n, m * k, ptr.data_ptr(), ci.data_ptr(), v.data_ptr(), lb.data_ptr(),
                                              ub.data_ptr(), 1e20, d.data_ptr(), d[m:].data_ptr(), c.data_ptr(),
                                              c[m:].data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms[k] = float(np.median(t[3:]))
    assert max(ms.values()) < 4 * ms[4097], ms
