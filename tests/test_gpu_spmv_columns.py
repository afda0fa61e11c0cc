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


def keeps_columns(S):
    u = S.weights_floats() // (32 * S.k)  # entries per lane
    return -(-S.k // 152) * u >= 16 * 24


@pytest.fixture(scope="module")
def matrix():
    rows, cols = W.rmat(scale=17, m_draws=1 << 21, seed=2)
    n = 1 << 17
    x0, w = W.spmv_inputs(n, rows.size, 2)
    return rows, cols, n, x0, w


@pytest.mark.parametrize("C,default_order", [(512, True), (300, True), (1024, True), (64, True), (5000, True), (512, False)])
def test_kept_columns(matrix, C, default_order):
    """The kernel with kept columns on both layouts, for other block sizes than the 512 its
    read-ahead is made for too."""
    rows, cols, n, x0, w = matrix
    S = E.Schedule.partition(rows, cols, n, C, bipartite=True, default_order=default_order)
    assert keeps_columns(S)
    check_both_layouts(S, rows, cols, x0, w, n)


def test_kept_columns_from_pinned_host_memory(matrix):
    rows, cols, n, x0, w = matrix
    S = E.Schedule.partition(rows, cols, n, 512, bipartite=True, default_order=True)
    assert keeps_columns(S)
    xh, wh = (torch.from_numpy(a.copy()).pin_memory() for a in (x0, w))
    yh = torch.full((n,), 3.0).pin_memory()
    for _ in range(2):
        S.run_host(xh, wh, yh, kernel=E.SPMV)
        check_field(yh, O.spmv(rows, cols, x0, w, n), "y")


@pytest.mark.parametrize("scale", [12, 17])
@pytest.mark.parametrize("shift", ["y starts in w", "w starts in y", "y is w's head"])
def test_result_over_the_weights(matrix, scale, shift):
    """y overlaps w: rows are written while weights are still read, so they go to a buffer
    of the schedule first."""
    if scale == 17:
        rows, cols, n, x0, w = matrix
    else:
        rows, cols = W.rmat(scale=scale, m_draws=1 << 16, seed=1)
        n = 1 << scale
        x0, w = W.spmv_inputs(n, rows.size, 0)
    S = E.Schedule.partition(rows, cols, n, 512, bipartite=True, default_order=True)
    m = rows.size
    buf = torch.empty(m + n, device="cuda")
    w_at, y_at = {"y starts in w": (0, m - 100), "w starts in y": (n - 100, 0), "y is w's head": (0, 0)}[shift]
    wd, y = buf[w_at:w_at + m], buf[y_at:y_at + n]
    wd.copy_(cuda(w))
    S.run(cuda(x0), wd, y, kernel=E.SPMV)
    check_field(y, O.spmv(rows, cols, x0, w, n), "y")
