"""The step kernels (flux_tma.cu) against the oracle, in schedule layout (GPU only).

Runs of several steps and gradients go to the resident kernels on most meshes,
so single steps are driven here call by call: every state width, stage counts,
in place and out of place, pending copies, self loops, repeated pairs and
blocks of one task.  Every test counts the edge launches (one per step) and asks
for the pipelined kernel's launch plan.
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
from parity import check_field, check_state  # noqa: E402


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.fixture(scope="module")
def mesh():
    src, dst = W.knn_mesh(4096, 4, 0)
    return src, dst, 4096


def edge_graph():
    rng = np.random.default_rng(4)
    src = rng.integers(0, 200, 777).astype(np.int32)
    dst = rng.integers(0, 200, 777).astype(np.int32)
    src[:20] = dst[:20]  # self loops
    src[20:40], dst[20:40] = src[40:60], dst[40:60]  # repeated pairs
    return src, dst, 300  # vertices from 200 on are untouched


def forward(S, src, dst, n, D, steps, seed, pending):
    x0, w, tau = W.flux_state(n, D, seed), W.flux_weights(src.size, seed), 1e-2
    assert S.pipeline_info(D)["grid"] > 0
    xl, yl = torch.zeros(S.layout_floats(D), device="cuda"), torch.zeros(S.layout_floats(D), device="cuda")
    ol, wl = torch.zeros_like(xl), torch.zeros(S.weights_floats(), device="cuda")
    S.layout_in(cuda(x0), xl)
    S.weights_in(cuda(w), wl)
    S.timing(2)
    for t in range(steps):
        if pending:
            S.step(D, xl, xl, wl, None, tau, pending=True)
        elif t % 2 == 0:  # out of place, back in place
            S.step(D, xl, yl, wl, ol, tau)
            xl, yl = yl, xl
        else:
            S.step(D, xl, xl, wl, ol, tau)
    if pending:
        S.finish(D, xl, tau)
    assert S.timing_read(E.T_EDGE_FWD)[1] == steps
    S.timing(0)
    x, out = torch.zeros(D, n, device="cuda"), torch.zeros(D, n, device="cuda")
    S.layout_out(xl, x)
    xT, fT = O.flux_steps(src, dst, x0, w, steps, tau)
    check_state(x, xT, x0, steps, "x")
    if not pending:
        S.layout_out(ol, out)
        check_field(out, fT, "out")
    assert S.check_errors() == 0


def adjoint(S, src, dst, n, D, steps, seed, pending):
    """Reverse steps at one state: lam_{t+1} = adjoint of a step at x0, weight gradients added up."""
    x0, w, g, tau = W.flux_state(n, D, seed), W.flux_weights(src.size, seed), W.loss_weights(n, D, seed), 1e-2
    assert S.pipeline_info(D, adjoint=True)["grid"] > 0
    xl, ll = torch.zeros(S.layout_floats(D), device="cuda"), torch.zeros(S.layout_floats(D), device="cuda")
    wl, gl = torch.zeros(S.weights_floats(), device="cuda"), torch.zeros(S.weights_floats(), device="cuda")
    S.layout_in(cuda(x0), xl)
    S.layout_in(cuda(g), ll)
    S.weights_in(cuda(w), wl)
    lam_ref, dw_ref = g.astype(np.float64), 0.0
    S.timing(2)
    for _ in range(steps):
        S.adjoint_step(D, xl, wl, ll, gl, tau, pending=pending)
        lam_ref, dw = O.flux_adjoint(src, dst, x0, w, 1, tau, lam_ref)
        dw_ref = dw_ref + dw
    if pending:
        S.adjoint_finish(D, ll, tau)
    assert S.timing_read(E.T_EDGE_ADJ)[1] == steps
    S.timing(0)
    lam, gw = torch.zeros(D, n, device="cuda"), torch.zeros(src.size, device="cuda")
    S.layout_out(ll, lam)
    S.weights_out_add(gl, gw)
    check_state(lam, lam_ref, g, steps, "lam")
    check_field(gw, dw_ref, "dw")
    assert S.check_errors() == 0


@pytest.mark.parametrize("pending", [False, True])
@pytest.mark.parametrize("stages", [2, 4])
@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 8])
def test_widths(mesh, D, stages, pending):
    src, dst, n = mesh
    S = E.Schedule.partition(src, dst, n, 256)
    S.set_pipeline(stages)
    forward(S, src, dst, n, D, 3, D, pending)
    adjoint(S, src, dst, n, D, 2, D, pending)


@pytest.mark.parametrize("default_order", [False, True])
@pytest.mark.parametrize("C", [1, 7, 100, 777, 5000])
def test_loops_pairs_and_tiny_blocks(C, default_order):
    src, dst, n = edge_graph()
    S = E.Schedule.partition(src, dst, n, C, default_order=default_order)
    for pending in (False, True):
        forward(S, src, dst, n, 5, 3, 2, pending)
        adjoint(S, src, dst, n, 5, 2, 2, pending)


@pytest.mark.parametrize("D", [1, 2, 3, 4, 6, 7, 8])
def test_one_step_run(mesh, D):
    src, dst, n = mesh
    S = E.Schedule.partition(src, dst, n, 256, default_order=D % 2 == 0)
    assert S.pipeline_info(D)["grid"] > 0
    x0, w = W.flux_state(n, D, 3), W.flux_weights(src.size, 3)
    x = cuda(x0)
    out = torch.zeros_like(x)
    S.timing(2)
    S.run(x, cuda(w), out, steps=1, tau=1e-2)
    assert S.timing_read(E.T_EDGE_FWD)[1] == 1
    xT, fT = O.flux_steps(src, dst, x0, w, 1, 1e-2)
    check_field(out, fT, "out")
    check_state(x, xT, x0, 1, "x")
    assert S.check_errors() == 0
