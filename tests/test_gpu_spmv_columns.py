"""SpMV with and without columns kept in shared memory, against the oracle (GPU only).

The kernel keeps columns where every SM has 24 blocks of 512 entries or more
(152 SMs: about 1.9M entries).
"""
import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1605_02043_gb300 as E  # noqa: E402
from parity import check_field  # noqa: E402


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def check_both_layouts(S, rows, cols, x0, w, n):
    ref = O.spmv(rows, cols, x0, w, n)
    y = torch.full((n,), 3.0, device="cuda")
    S.run(cuda(x0), cuda(w), y, kernel=E.SPMV)
    check_field(y, ref, "y")
    xl, wl = torch.empty(n, device="cuda"), torch.empty(S.weights_floats(), device="cuda")
    yl, y2 = torch.full((n,), 5.0, device="cuda"), torch.empty(n, device="cuda")
    S.spmv_x_in(cuda(x0), xl)
    S.weights_in(cuda(w), wl)
    S.spmv(xl, wl, yl)
    S.spmv_y_out(yl, y2)
    check_field(y2, ref, "y (layout entry points)")
    assert S.check_errors() == 0


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7])
def test_few_columns_many_entries(n):
    """Enough entries for the kept columns, but fewer than four columns to keep (16
    bytes).  Positive values: a row sums up to 2M products without cancellation."""
    m = 2_000_003
    rng = np.random.default_rng(n)
    rows, cols = (np.sort(rng.integers(0, n, m)).astype(np.int32), rng.integers(0, n, m).astype(np.int32))
    x0, w = (rng.uniform(0.5, 1.5, n).astype(np.float32), rng.uniform(0, 1, m).astype(np.float32))
    S = E.Schedule.partition(rows, cols, n, 512, bipartite=True, default_order=True)
    check_both_layouts(S, rows, cols, x0, w, n)
