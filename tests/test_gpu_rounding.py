"""Rounding of the interaction d / (1 + |d|^2) in every edge kernel (GPU only).

A matching (every vertex in one task, weight 1) of close states, |d_c| ~ 0.1 as
on a smooth field: each result is one term, so its error is the term's own.  The
states are multiples of 2^-20, so d is exact.  What an FP32 term may be off,
relative rms against 64 bits: the denominator 1 + |d|^2 rounded once at a value
in [1, 2) (uniform within 2^-24: 3.4e-8), its reciprocal off by up to 1 ulp
(2^-24 at a value near 0.9: 4.0e-8 if uniform), the product rounded once (at
most 3.4e-8, mean over the binade 2.5e-8): 5.8e-8 together.  Summing |d|^2 onto
1 instead rounds D times at that size: 7.6e-8 at D = 5 and 9.4e-8 at D = 8 with
an exact reciprocal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1605_02043_gb300 as E  # noqa: E402

BOUND = 6e-8
PAIRS = 1 << 15


def matching(D, seed):
    rng = np.random.default_rng(seed)
    n = 2 * PAIRS
    perm = rng.permutation(n).astype(np.int32)
    x = np.round(rng.normal(0, 0.1 / np.sqrt(2), (D, n)) * 2.0 ** 20) / 2.0 ** 20
    src, dst = perm[0::2].copy(), perm[1::2].copy()
    d = x[:, dst] - x[:, src]
    term = d / (1 + (d * d).sum(0))
    S = E.Schedule.partition(src, dst, n, 512, default_order=True)
    return S, src, dst, torch.from_numpy(x.astype(np.float32)).cuda(), d, term


def rms(got, ref):
    got = np.asarray(got.detach().cpu().numpy(), np.float64)
    ok = ref != 0
    return float(np.sqrt(np.mean(((got - ref)[ok] / ref[ok]) ** 2)))


@pytest.mark.parametrize("D", [1, 5, 8])
@pytest.mark.parametrize("path", ["run", "pipelined", "one block", "read-only"])
def test_forward_term(D, path):
    S, src, dst, x, _, term = matching(D, D)
    w, out = torch.ones(PAIRS, device="cuda"), torch.empty_like(x)
    if path == "one block":
        S.set_pipeline(0)
    if path == "read-only":
        S.set_cache(E.CACHE_L1)
    S.timing(2)
    # two steps of length 0 are one launch of the resident kernel
    S.run(x, w, out, steps=2 if path == "run" else 1, tau=0.0)
    assert S.timing_read(E.T_EDGE_FWD)[1] == 1
    assert rms(out[:, torch.from_numpy(src).cuda().long()], term) <= BOUND
    assert rms(out[:, torch.from_numpy(dst).cuda().long()], -term) <= BOUND
    assert S.check_errors() == 0


@pytest.mark.parametrize("D", [1, 5, 8])
@pytest.mark.parametrize("path", ["run", "pipelined", "one block"])
def test_adjoint_term(D, path):
    # a cotangent of one component at the first endpoints: the weight gradient
    # of a step of length 1 is -d_0 / (1 + |d|^2)
    S, src, dst, x, d, term = matching(D, D + 10)
    w = torch.ones(PAIRS, device="cuda")
    lam = torch.zeros_like(x)
    lam[0, torch.from_numpy(src).cuda().long()] = 1.0
    gw = torch.zeros(PAIRS, device="cuda")
    if path == "pipelined":
        f32 = dict(device="cuda")
        xl, ll = torch.zeros(S.layout_floats(D), **f32), torch.zeros(S.layout_floats(D), **f32)
        wl, gl = torch.zeros(S.weights_floats(), **f32), torch.zeros(S.weights_floats(), **f32)
        S.layout_in(x, xl)
        S.layout_in(lam, ll)
        S.weights_in(w, wl)
        S.adjoint_step(D, xl, wl, ll, gl, tau=1.0)
        S.weights_out_add(gl, gw)
    else:
        if path == "one block":
            S.set_pipeline(0)
        S.run_adjoint(x, w, lam, gw, steps=1, tau=1.0)
    assert rms(gw.abs(), np.abs(term[0])) <= BOUND
    assert S.check_errors() == 0
