"""What a program has this library do, as cases that can be timed and checked.

Explicit time stepping of a node state over an unstructured mesh (the flux
kernel), its gradient for fitting, and y = A x on a power-law matrix, each
through the public Python calls: single steps and loops in schedule layout,
whole runs in the caller's layout, the autograd function, the graph-captured
runner over a batch of meshes, SpMV in both layouts and the host-buffer call.

A case is a dict: `kind` names the calls, `n` the mesh nodes (or matrix rows),
`C` the tasks per block, `D` the state width, `steps` the explicit steps of
one pass, `order` the task order ("partitioned", or "default" for the input
order).  Graphs, states and weights are all drawn from the seed, on the GPU:
meshes join every point of a uniform cloud to its 4 nearest (the bench's
mesh), matrices are R-MAT (a, b, c, d = 0.57, 0.19, 0.19, 0.05) with 16 draws
per row in CSR order.
"""
import math

import numpy as np
import torch

import paper_1605_02043_gb300 as ep
from paper_1605_02043_gb300.autograd import FluxRunner, flux_steps

TAU = 2.0 ** -10  # the same number in 32 and 64 bits
DEV = "cuda"


def _flux(kind, n, C, D, steps, order="partitioned", **more):
    return dict(kind=kind, n=n, C=C, D=D, steps=steps, order=order, **more)


def listed():
    return [
        # the smallest call: one complete step with its flux on a small mesh,
        # as a program that looks at the state after every step makes it
        dict(name="step_4k", **_flux("step", 4096, 256, 5, 1)),
        # the bench's mesh, ten steps issued one by one with the shared copies
        # pending (a solver that keeps its state in schedule layout and adapts
        # something between steps), finished and read out
        dict(name="loop_1m", **_flux("loop", 1 << 20, 512, 5, 10)),
        # the largest: a long run of the bench's mesh in one call
        dict(name="run_1m", **_flux("run", 1 << 20, 512, 5, 100)),
        # an ordinary mesh of odd size, a run of some length
        dict(name="run_64k", **_flux("run", 65521, 512, 5, 50)),
        # a scalar field (heat, concentration), short run
        dict(name="run_400k_d1", **_flux("run", 400009, 512, 1, 20)),
        # the widest state, ragged size, the large blocks of the paper's sweep
        dict(name="run_150k_d8", **_flux("run", 150001, 1024, 8, 10)),
        # the input order, which runs while the partition is still being made
        dict(name="run_256k_default", **_flux("run", 1 << 18, 512, 5, 10, "default")),
        # gradients of a ten-step run for the state and the weights, eager
        dict(name="train_256k", **_flux("train", 1 << 18, 512, 5, 10, every=5)),
        # many uneven meshes in one schedule, forward and backward replayed
        # from a CUDA graph with new inputs every pass
        dict(name="train_batch", **_flux("batch", 32768, 1024, 5, 20, every=10, meshes=32)),
        # y = A x with the weights kept in schedule layout (an iterative
        # solver), CSR order
        dict(name="spmv_1m_csr", kind="spmv", n=1 << 20, C=512, order="default"),
        # y = A x in the caller's layout with new weights, partitioned order
        dict(name="spmv_256k", kind="spmv_run", n=1 << 18, C=512, order="partitioned"),
        # the flux of a state in pinned host memory (a solver on the host)
        dict(name="host_256k", **_flux("host", 1 << 18, 512, 5, 1)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "loop", "run", "run", "run", "train", "batch", "spmv", "spmv_run", "host"])
    C = rng.choice([256, 512, 512, 768, 1024])
    order = rng.choice(["partitioned", "partitioned", "partitioned", "default"])
    if kind in ("spmv", "spmv_run"):
        return dict(kind=kind, n=1 << rng.randint(12, 18), C=C, order=order)
    D = rng.choice([1, 2, 3, 4, 5, 5, 5, 6, 7, 8])
    if kind == "step":
        return _flux(kind, _log_int(rng, 1024, 1 << 20), C, D, 1, order)
    if kind == "loop":
        return _flux(kind, _log_int(rng, 1024, 1 << 20), C, D, rng.randint(2, 20), order)
    if kind == "run":
        return _flux(kind, _log_int(rng, 1024, 700000), C, D, _log_int(rng, 1, 100), order)
    if kind == "train":
        return _flux(kind, _log_int(rng, 1024, 1 << 18), C, D, rng.randint(2, 16), order, every=rng.randint(1, 8))
    if kind == "batch":
        return _flux(kind, _log_int(rng, 2048, 32768), C, D, rng.randint(4, 24), order, every=rng.randint(2, 10),
                     meshes=rng.randint(2, 40))
    return _flux(kind, _log_int(rng, 1024, 1 << 19), C, D, 1, order)


# ---------------------------------------------------------------------- inputs


def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + stream)


def _mesh(n, gen, k=4):
    """(src, dst) of the k-nearest-neighbour mesh of n uniform points, each pair
    once, in random order (neighbours looked for in the 27 cells around)."""
    p = torch.rand(n, 3, device=DEV, generator=gen)
    g = max(1, int((n / 3) ** (1 / 3)))
    c = (p * g).long().clamp_(max=g - 1)
    cell = (c[:, 0] * g + c[:, 1]) * g + c[:, 2]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=g ** 3)
    start = count.cumsum(0) - count
    cap = int(count.max())
    table = torch.full((g ** 3, cap), -1, dtype=torch.int64, device=DEV)
    sc = cell[order]
    table[sc, torch.arange(n, device=DEV) - start[sc]] = order
    r = torch.arange(-1, 2, device=DEV)
    off = torch.cartesian_prod(r, r, r)
    key = []
    for i in range(0, n, 1 << 16):
        q = torch.arange(i, min(n, i + (1 << 16)), device=DEV)
        nb = c[q][:, None, :] + off[None]
        inside = ((nb >= 0) & (nb < g)).all(-1)
        nb = nb.clamp(0, g - 1)
        cand = table[(nb[..., 0] * g + nb[..., 1]) * g + nb[..., 2]]
        cand = torch.where(inside[..., None], cand, -1).flatten(1)
        d = (p[cand.clamp(min=0)] - p[q][:, None]).square_().sum(-1)
        d = torch.where((cand < 0) | (cand == q[:, None]), math.inf, d)
        near, at = d.topk(min(k, d.shape[1]), largest=False)
        b = cand.gather(1, at)
        a = q[:, None].expand_as(b)
        ok = near < math.inf
        a, b = a[ok], b[ok]
        key.append(torch.minimum(a, b) * n + torch.maximum(a, b))
    key = torch.unique(torch.cat(key))
    key = key[torch.randperm(key.numel(), device=DEV, generator=gen)][:_tasks(n)]
    return (key // n).int(), (key % n).int()


def _tasks(n):
    """Tasks of a mesh of n nodes: about 98% of the pairs found, a fixed number so
    that every seed's gradients have the same shape."""
    return 12 * n // 5


def _rmat(n, gen):
    """(rows, cols) of an R-MAT matrix of n rows (a power of two), CSR order."""
    m = 16 * n
    row = torch.zeros(m, dtype=torch.int64, device=DEV)
    col = torch.zeros_like(row)
    for _ in range(n.bit_length() - 1):
        u = torch.rand(m, device=DEV, generator=gen)
        row = 2 * row + (u >= 0.76)
        col = 2 * col + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    keep = row != col
    key = torch.unique(row[keep] * n + col[keep])
    return (key // n).int(), (key % n).int()


def _batch_sizes(case):
    """Nodes of a batch's meshes, log-uniform in [1024, n]."""
    u = np.random.default_rng(case["meshes"]).random(case["meshes"])
    return np.rint(1024 * (case["n"] / 1024) ** u).astype(int).tolist()


def _graphs(case, seed):
    """List of (nodes, src, dst), device tensors: one graph, or a batch's meshes."""
    gen = _gen(seed, 1)
    n = case["n"]
    if case["kind"] in ("spmv", "spmv_run"):
        return [(n, *_rmat(n, gen))]
    if case["kind"] != "batch":
        return [(n, *_mesh(n, gen))]
    return [(s, *_mesh(s, gen)) for s in _batch_sizes(case)]


def _union(graphs):
    src, dst, n = [], [], 0
    for nodes, s, d in graphs:
        src.append(s + n)
        dst.append(d + n)
        n += nodes
    return n, torch.cat(src), torch.cat(dst)


def _fields(case, seed, n, m):
    """x, w and the loss cotangent g (None where the case has no gradient)."""
    gen = _gen(seed, 2)
    if case["kind"] in ("spmv", "spmv_run"):
        return 2 * torch.rand(n, device=DEV, generator=gen) - 1, torch.rand(m, device=DEV, generator=gen), None
    x = torch.randn(case["D"], n, device=DEV, generator=gen)
    w = 0.5 + torch.rand(m, device=DEV, generator=gen)
    return x, w, torch.randn(case["D"], n, device=DEV, generator=gen)


def _schedule(graph, case, threads=0):
    n, src, dst = graph
    return ep.Schedule.partition(src.cpu().numpy(), dst.cpu().numpy(), n, case["C"],
                                 bipartite=case["kind"] in ("spmv", "spmv_run"),
                                 default_order=case["order"] == "default", threads=threads)


def prepare(case, seed):
    graphs = _graphs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        S = ep.Schedule.batch([_schedule(g, case) for g in graphs])
    else:
        S = _schedule(graphs[0], case)
    x, w, g = _fields(case, seed, S.n, S.m)
    s = dict(case=case, S=S, x=x, w=w, g=g)
    D = case.get("D", 1)
    if kind in ("step", "loop"):
        s["x_lay"] = torch.empty(S.layout_floats(D), device=DEV)
        s["x2_lay"] = torch.empty_like(s["x_lay"])
        s["out_lay"] = torch.empty_like(s["x_lay"])
        s["w_lay"] = torch.empty(S.weights_floats(), device=DEV)
        S.layout_in(x, s["x_lay"])
        S.weights_in(w, s["w_lay"])
    elif kind == "spmv":
        s["x_lay"] = torch.empty(S.n, device=DEV)
        s["y_lay"] = torch.empty(S.n, device=DEV)
        s["w_lay"] = torch.empty(S.weights_floats(), device=DEV)
        S.weights_in(w, s["w_lay"])
    elif kind == "batch":
        R = FluxRunner(S, D, case["steps"], TAU, case["every"])
        R.load(x, w, g)
        R.run()
        torch.cuda.synchronize()
        s["runner"], s["graph"] = R, torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            R.run()
    elif kind == "host":
        s["x"], s["w"] = x.cpu().pin_memory(), w.cpu().pin_memory()
        s["out"] = torch.empty_like(s["x"]).pin_memory()
    return s


# ------------------------------------------------------------------------ runs


def run(state):
    case, S, x, w = state["case"], state["S"], state["x"], state["w"]
    kind, D, steps = case["kind"], case.get("D", 1), case.get("steps", 1)
    if kind == "step":
        S.step(D, state["x_lay"], state["x2_lay"], state["w_lay"], state["out_lay"], TAU)
        x1, f = torch.empty_like(x), torch.empty_like(x)
        S.layout_out(state["x2_lay"], x1)
        S.layout_out(state["out_lay"], f)
        return x1, f
    if kind == "loop":
        xl = state["x2_lay"]
        S.step(D, state["x_lay"], xl, state["w_lay"], None, TAU, pending=True)
        for _ in range(steps - 1):
            S.step(D, xl, xl, state["w_lay"], None, TAU, pending=True)
        S.finish(D, xl, TAU)
        xT = torch.empty_like(x)
        S.layout_out(xl, xT)
        return xT
    if kind == "run":
        xT, f = x.clone(), torch.empty_like(x)
        S.run(xT, w, f, steps=steps, tau=TAU)
        return xT, f
    if kind == "train":
        x, w = x.detach().requires_grad_(), w.detach().requires_grad_()
        xT = flux_steps(x, w, S, steps, TAU, case["every"])
        dx, dw = torch.autograd.grad(xT, (x, w), state["g"])
        return xT.detach(), dx, dw
    if kind == "batch":
        state["runner"].load(x, w, state["g"])
        state["graph"].replay()
        return state["runner"].results(x, S.m)
    if kind == "spmv":
        y = torch.empty_like(x)
        S.spmv_x_in(x, state["x_lay"])
        S.spmv(state["x_lay"], state["w_lay"], state["y_lay"])
        S.spmv_y_out(state["y_lay"], y)
        return y
    if kind == "spmv_run":
        y = torch.empty_like(x)
        S.run(x, w, y, kernel=ep.SPMV)
        return y
    S.run_host(x, w, state["out"], steps=1, tau=0.0, D=D)  # tau 0: x stays, out is its flux
    return state["out"]


# -------------------------------------------------------------- work and truth


def _sizes(case):
    """Nodes and tasks (a matrix's entries: what its duplicates leave on average)."""
    n = case["n"]
    if case["kind"] in ("spmv", "spmv_run"):
        left = {12: 0.82, 13: 0.85, 14: 0.87, 15: 0.89, 16: 0.91, 17: 0.925, 18: 0.94}
        return n, round(16 * n * left.get(n.bit_length() - 1, 0.95))
    sizes = _batch_sizes(case) if case["kind"] == "batch" else [n]
    return sum(sizes), sum(_tasks(s) for s in sizes)


def work(case):
    n, m = _sizes(case)
    kind, D, steps = case["kind"], case.get("D", 1), case.get("steps", 1)
    task = 8 + 4  # two vertex ids and the weight
    if kind in ("spmv", "spmv_run"):
        return dict(bytes=task * m + 8 * n, flops=2 * m)
    flux = (5 * D + 4) * m  # difference, its square, the division, two scatters
    if kind in ("train", "batch"):
        # x, g in; xT, dL/dx out; the weight gradient out; forward, and the
        # reverse step's products at every state
        return dict(bytes=(task + 4) * m + 16 * D * n, flops=steps * (flux + (10 * D + 8) * m))
    states = {"step": 3, "loop": 2, "run": 3, "host": 2}[kind]
    return dict(bytes=task * m + 4 * D * n * states, flops=steps * flux)


def _flux64(x, w, src, dst):
    d = x[:, dst] - x[:, src]
    f = w * d / (1 + (d * d).sum(0))
    return torch.zeros_like(x).index_add(1, src, f).index_add(1, dst, -f)


def exact(case, seed):
    n, src, dst = _union(_graphs(case, seed))
    src, dst = src.long(), dst.long()
    x, w, g = (None if t is None else t.double() for t in _fields(case, seed, n, src.numel()))
    kind, steps = case["kind"], case.get("steps", 1)
    if kind in ("spmv", "spmv_run"):
        return torch.zeros_like(x).index_add(0, src, w * x[dst])
    if kind == "host":
        return _flux64(x, w, src, dst)
    if kind in ("train", "batch"):
        x, w = x.requires_grad_(), w.requires_grad_()
        xT = x
        for _ in range(steps):
            xT = xT + TAU * _flux64(xT, w, src, dst)
        dx, dw = torch.autograd.grad(xT, (x, w), g)
        return xT.detach(), dx, dw
    f = None
    for _ in range(steps):
        f = _flux64(x, w, src, dst)
        x = x + TAU * f
    return x if kind == "loop" else (x, f)
