"""Resident runs of several steps (march.cu) against the oracle (GPU only).

Sizes where the layout has its edges: one part, parts of a few vertices, the
last slice partly filled, a halo larger than the part (default order), slots
kept in shared memory and slots read from the L2, every state width, isolated
vertices, self loops and repeated pairs.  Tolerances: parity.py.
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
from paper_1605_02043_gb300._lib import EpError  # noqa: E402
from parity import check_field, check_state  # noqa: E402


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def run_against_oracle(S, src, dst, n, D, steps, seed, tau=1e-2):
    x0, w = W.flux_state(n, D, seed), W.flux_weights(src.size, seed)
    x = cuda(x0)
    out = torch.full_like(x, 7.0)
    S.timing(2)
    S.run(x, cuda(w), out, steps=steps, tau=tau)
    launches = S.timing_read(E.T_EDGE_FWD)[1]
    S.timing(0)
    assert S.check_errors() == 0
    xT, fT = O.flux_steps(src, dst, x0, w, steps, tau)
    check_field(out, fT, "out")
    check_state(x, xT, x0, steps, "x")
    return launches


@pytest.mark.parametrize("n,C,D,steps,default_order", [
    (40, 16, 5, 3, False), (129, 64, 1, 2, False), (300, 64, 5, 9, True), (1025, 256, 3, 4, False),
    (4096, 256, 2, 5, False), (4096, 1000, 4, 5, True), (9999, 512, 6, 3, False), (9999, 512, 7, 4, True),
    (20011, 512, 8, 3, False), (50021, 1024, 5, 6, False), (50021, 512, 5, 2, True), (200003, 512, 1, 3, False),
])
def test_runs_match_oracle(n, C, D, steps, default_order):
    src, dst = W.knn_mesh(n, 4, 1)
    S = E.Schedule.partition(src, dst, n, C, default_order=default_order)
    assert run_against_oracle(S, src, dst, n, D, steps, n) == 1  # one launch for the whole run
    # again on the same schedule: the step counters go on from where they stand
    assert run_against_oracle(S, src, dst, n, D, steps + 1, n + 1) == 1


def test_slots_in_shared_memory_and_from_l2():
    # widths from 1 to 8 on one mesh: with D = 1 a part's slots fit beside its
    # state, with D = 8 they do not
    n = 320000
    src, dst = W.knn_mesh(n, 4, 2)
    S = E.Schedule.partition(src, dst, n, 1024)
    for D in (1, 5, 8):
        assert run_against_oracle(S, src, dst, n, D, 2, D) == 1


def test_loops_pairs_and_isolated_vertices():
    rng = np.random.default_rng(4)
    n = 3000
    src = rng.integers(0, 2000, 7777).astype(np.int32)
    dst = ((src + rng.integers(1, 30, 7777)) % 2000).astype(np.int32)
    src[:50] = dst[:50]
    src[50:100], dst[50:100] = src[100:150], dst[100:150]
    S = E.Schedule.partition(src, dst, n, 100)
    assert run_against_oracle(S, src, dst, n, 5, 4, 3) == 1


def test_hub_takes_the_step_kernels():
    # one vertex in every task: its slots would be one lane's
    n = 2000
    src, dst = np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32)
    S = E.Schedule.partition(src, dst, n, 128)
    assert run_against_oracle(S, src, dst, n, 3, 3, 3, tau=1e-4) == 3


@pytest.mark.parametrize("n,C,D,steps,every,default_order", [
    (40, 16, 5, 3, 2, False), (129, 64, 1, 1, 1, False), (300, 64, 3, 7, 3, True), (4096, 256, 2, 6, 6, False),
    (9999, 512, 5, 10, 1, False), (20011, 512, 8, 4, 3, False), (50021, 1024, 5, 5, 9, False),
    (9999, 512, 6, 2, 2, True), (120011, 512, 4, 5, 2, False), (200003, 1024, 7, 3, 5, False),
])
def test_gradients_match_oracle(n, C, D, steps, every, default_order):
    """Forward run and reverse sweep in one launch each (autograd and ep_run_adjoint);
    isolated vertices keep their state and cotangent."""
    from paper_1605_02043_gb300.autograd import flux_steps

    src, dst = W.knn_mesh(n, 4, 1)
    n += 3  # untouched
    S = E.Schedule.partition(src, dst, n, C, default_order=default_order)
    assert S.grad_sizes(D)[0] > 0
    x0, w, g, tau = W.flux_state(n, D, n), W.flux_weights(src.size, n), W.loss_weights(n, D, 1), 1e-2
    xT_ref, _ = O.flux_steps(src, dst, x0, w, steps, tau)
    dx_ref, dw_ref = O.flux_adjoint(src, dst, x0, w, steps, tau, g)
    for _ in range(2):
        x, wt = cuda(x0).requires_grad_(True), cuda(w).requires_grad_(True)
        S.timing(2)
        xT = flux_steps(x, wt, S, steps, tau, every)
        xT.backward(cuda(g))
        assert (S.timing_read(E.T_EDGE_FWD)[1], S.timing_read(E.T_EDGE_ADJ)[1]) == (1, 1)
        S.timing(0)
        check_state(xT, xT_ref, x0, steps, "xT")
        check_state(x.grad, dx_ref, g, steps, "dx0")
        check_field(wt.grad, dw_ref, "dw")
    lam, gw = cuda(g), torch.full((src.size,), 2.0, device="cuda")
    S.run_adjoint(cuda(x0), cuda(w), lam, gw, steps=steps, tau=tau)
    check_state(lam, dx_ref, g, steps, "dx0 (ep_run_adjoint)")
    check_field(gw, 2.0 + dw_ref, "accumulated dw (ep_run_adjoint)")
    assert S.check_errors() == 0


def test_two_streams_and_graph_replay():
    """Runs of two schedules on two streams, then captured and replayed."""
    n = 30011
    src, dst = W.knn_mesh(n, 4, 5)
    Ss = [E.Schedule.partition(src, dst, n, C) for C in (256, 512)]
    x0, w = W.flux_state(n, 5, 1), W.flux_weights(src.size, 1)
    xT, _ = O.flux_steps(src, dst, x0, w, 20, 1e-3)
    streams = [torch.cuda.Stream() for _ in Ss]
    wd, xs = cuda(w), [cuda(x0) for _ in Ss]
    torch.cuda.synchronize()
    for _ in range(2):
        for S, st, x in zip(Ss, streams, xs):
            with torch.cuda.stream(st):
                S.run(x, wd, None, steps=10, tau=1e-3)
    torch.cuda.synchronize()
    for S, x in zip(Ss, xs):
        assert S.check_errors() == 0
        check_state(x, xT, x0, 20, "x")
    x = cuda(x0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        Ss[0].run(x, wd, None, steps=5, tau=1e-3)
    for _ in range(4):
        g.replay()
    torch.cuda.synchronize()
    assert Ss[0].check_errors() == 0
    check_state(x, xT, x0, 20, "x (graph)")


def test_wait_for_a_neighbour_expires_then_recovers():
    """Part 0 leaves after its first published step (ep_debug_stall): the others' bounded
    wait runs out, the error is reported, and the next run is correct."""
    n = 30011
    src, dst = W.knn_mesh(n, 4, 5)
    S = E.Schedule.partition(src, dst, n, 512)
    x0, w = W.flux_state(n, 5, 2), W.flux_weights(src.size, 2)
    S.debug_stall(1)
    S.run(cuda(x0), cuda(w), None, steps=4, tau=1e-3)
    with pytest.raises(EpError) as ei:
        S.check_errors()
    assert ei.value.code == -4
    S.debug_stall(-1)
    assert run_against_oracle(S, src, dst, n, 5, 4, 2, tau=1e-3) == 1


@pytest.mark.parametrize("n,D,steps,every", [(131072, 8, 6, 1), (131072, 5, 6, 1), (90001, 8, 7, 2), (4099, 8, 9, 1)])
def test_checkpoints_hold_one_state_each(n, D, steps, every):
    """Every checkpoint of a forward run is the state before its step, own records and
    halo: the copy out of shared memory must be over before the next state overwrites
    it.  Input order: images several times a part's own records beside few slices, so
    the copy has the least time."""
    src, dst = W.knn_mesh(n, 4, 6)
    S = E.Schedule.partition(src, dst, n, 512, default_order=True)
    ns, nw = S.grad_sizes(D)
    assert ns > 0
    x0, w, tau = W.flux_state(n, D, 6), W.flux_weights(src.size, 6), 1e-2
    f32 = dict(device="cuda", dtype=torch.float32)
    x, wl = cuda(x0), torch.empty(nw, **f32)
    xl, xT = torch.empty(ns, **f32), torch.empty(ns, **f32)
    S.grad_state_in(x, xl)
    S.grad_weights_in(D, cuda(w), wl)
    nseg = -(-steps // every)
    ref = [x0.astype(np.float64)]
    for _ in range(nseg - 1):
        ref.append(O.flux_steps(src, dst, ref[-1], w, every, tau)[0])
    got = torch.empty_like(x)
    for _ in range(5):
        ckpt = torch.full((nseg, ns), float("nan"), **f32)
        S.grad_forward(D, xl, xT, wl, ckpt, steps, every, tau)
        for i in range(nseg):
            S.grad_state_out(ckpt[i], got)
            check_state(got, ref[i], x0, i * every, f"checkpoint {i}")
    # the halo parts of the images are what the reverse sweep recomputes from
    g = W.loss_weights(n, D, 2)
    lam, gw, work = torch.empty(ns, **f32), torch.empty(nw, **f32), torch.empty(max(every, 2) * ns, **f32)
    gl = torch.empty(ns, **f32)
    S.grad_state_in(cuda(g), gl)
    S.grad_backward(D, ckpt, work, wl, gl, lam, gw, steps, every, tau)
    S.grad_state_out(lam, got)
    dw = torch.empty(src.size, **f32)
    S.grad_weights_out(D, gw, dw)
    dx_ref, dw_ref = O.flux_adjoint(src, dst, x0, w, steps, tau, g)
    check_state(got, dx_ref, g, steps, "dx0")
    check_field(dw, dw_ref, "dw")
    assert S.check_errors() == 0


def test_single_steps_make_no_resident_layout():
    """One-step runs and single steps allocate nothing for resident runs; the first run of
    several steps does (a state and the weights at the least)."""
    n, D = 200003, 5
    src, dst = W.knn_mesh(n, 4, 8)
    S = E.Schedule.partition(src, dst, n, 512)
    x0, w = W.flux_state(n, D, 8), W.flux_weights(src.size, 8)
    x, wd = cuda(x0), cuda(w)
    out = torch.zeros_like(x)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    S.run(x, wd, out, steps=1, tau=1e-2)
    before = free()
    for _ in range(2):
        S.run(x, wd, out, steps=1, tau=1e-2)
    assert free() == before
    S.run(x, wd, out, steps=2, tau=1e-2)
    after = free()
    ns, nw = S.grad_sizes(D)
    assert before - after >= 4 * (ns + nw)
    xT, fT = O.flux_steps(src, dst, x0, w, 5, 1e-2)
    check_state(x, xT, x0, 5, "x")
    check_field(out, fT, "out")


def test_run_captured_before_any_eager_one():
    """A run of several steps captured after single steps only: nothing can be allocated or
    uploaded there, so it takes the step kernels; captured again after an eager run."""
    n, D = 30011, 5
    src, dst = W.knn_mesh(n, 4, 9)
    S = E.Schedule.partition(src, dst, n, 512)
    x0, w = W.flux_state(n, D, 9), W.flux_weights(src.size, 9)
    x, wd = cuda(x0), cuda(w)
    out = torch.zeros_like(x)
    S.run(x, wd, out, steps=1, tau=1e-3)
    for eager in (False, True):
        if eager:
            S.run(x, wd, out, steps=4, tau=1e-3)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            S.run(x, wd, out, steps=4, tau=1e-3)
        x.copy_(cuda(x0))
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        xT, fT = O.flux_steps(src, dst, x0, w, 12, 1e-3)
        check_state(x, xT, x0, 12, "x")
        check_field(out, fT, "out")
    assert S.check_errors() == 0


SMEM = 227 * 1024 - 512  # what a block of the resident kernels may ask for


def slots_from_l2(S, D, grad):
    """True where a part cannot keep its slots and weights in shared memory beside its
    state (and cotangent): the mean part's need is above the limit, so the largest's is.
    A state has D floats a record, a weight buffer 64 a column (entries and weights 384 bytes)."""
    ns, nw = S.grad_sizes(1)
    assert ns > 0 and S.n >= 152 * 64  # 152 parts
    return (2 if grad else 1) * 4 * D * ns / 152 + 384 * nw / 64 / 152 > SMEM


@pytest.fixture(scope="module")
def large_mesh():
    """(n, default order) -> (src, dst, schedule), one mesh kept at a time."""
    kept = {}

    def get(n, default_order):
        if (n, default_order) not in kept:
            kept.clear()
            src, dst = W.knn_mesh(n, 4, 2)
            kept[n, default_order] = src, dst, E.Schedule.partition(src, dst, n, 1024, default_order=default_order)
        return kept[n, default_order]

    yield get
    kept.clear()


# the forward kernel's variants: 512 threads (D = 5 in input order), 1024 (more
# than 128 slices a part) and the widths with one thread count; g: gradients; r: the
# mean part fits, so slots stay in shared memory with 1024 threads (D = 3) and 512
@pytest.mark.parametrize("n,default_order,what", [
    (400001, True, "f5"), (400001, False, "g6"), (520001, False, "f7 f8 g4 g5"), (640001, False, "r3 f5 f6 g3"),
    (1 << 20, False, "f1 f2 f3 f4 g1 g2"), (320000, False, "r5 g8"),
])
def test_slots_read_from_the_l2(large_mesh, n, default_order, what):
    from paper_1605_02043_gb300.autograd import flux_steps

    src, dst, S = large_mesh(n, default_order)
    w = W.flux_weights(src.size, 1)
    for kind, D in ((k[0], int(k[1])) for k in what.split()):
        assert slots_from_l2(S, D, kind == "g") == (kind != "r")
        if kind != "g":
            assert run_against_oracle(S, src, dst, n, D, 2, D) == 1
            continue
        assert S.grad_sizes(D)[0] > 0
        x0, g, tau = W.flux_state(n, D, D), W.loss_weights(n, D, 1), 1e-2
        x, wt = cuda(x0).requires_grad_(True), cuda(w).requires_grad_(True)
        xT = flux_steps(x, wt, S, 3, tau, 2)
        xT.backward(cuda(g))
        dx_ref, dw_ref = O.flux_adjoint(src, dst, x0, w, 3, tau, g)
        check_state(x.grad, dx_ref, g, 3, f"dx0 D={D}")
        check_field(wt.grad, dw_ref, f"dw D={D}")
    assert S.check_errors() == 0
