"""GPU: the final bound where sums and terms leave the middle of FP32's range.

The sums g = W^T rho are formed on FP32 levels and the error bounds in FP32;
what those cannot hold is formed in FP64, so the bound stays within 1e-11 of
the terms' size (FP64 sums of at most 3000 terms carry about 3e-13) and at most
1e-12 of it above the FP64 oracle's q, at duals of size 1 as at 1e36 (sums
beyond 2^117), at bounds that make the terms larger than any FP32 number, and on
a net whose every term is about 1e-25.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import outward_f32

pytestmark = pytest.mark.gpu

# input shape, convs (cout, k, stride, pad) with a blocked and a general transposed pass, FC widths
NETS = {
    "fc": ((40,), [], [130, 65, 1]),
    "conv": ((3, 12, 12), [(8, 4, 2, 1), (12, 3, 1, 1), (6, 5, 1, 2)], [33, 1]),
    "channels": ((4, 6, 6), [(80, 3, 1, 1), (8, 4, 2, 1), (130, 3, 1, 1)], [9, 1]),  # more than a block of output channels
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


def _problem(name, dual, bound=1.0, last=1.0, zero_rows=False, B=4):
    """Net, box, bounds and duals: duals of size `dual`, intermediate bounds widened by `bound`, W_n scaled by `last`."""
    shape, convs, fcs = NETS[name]
    rng = np.random.default_rng(17)
    n0 = int(np.prod(shape))
    c0 = rng.uniform(-0.5, 0.5, n0)
    specs = []
    for cout, k, s, p in convs:
        W = rng.normal(0, np.sqrt(2 / (shape[0] * k * k)), (cout, shape[0], k, k)).astype(np.float32)
        specs.append(synth.LayerSpec("conv", W, rng.normal(0, 0.1, cout).astype(np.float32), shape, s, p))
        shape = specs[-1].out_shape
    n = int(np.prod(shape))
    for m in fcs:
        specs.append(synth.LayerSpec("fc", rng.normal(0, np.sqrt(2 / n), (m, n)).astype(np.float32),
                                     rng.normal(0, 0.1, m).astype(np.float32), (n,)))
        n = m
    top = specs[-1]
    specs[-1] = synth.LayerSpec("fc", top.W * np.float32(last), top.b * np.float32(0 if last != 1 else 1), top.in_shape)
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
                     oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs])
    l0, u0 = (c0 - 0.05).astype(np.float32)[None], (c0 + 0.05).astype(np.float32)[None]
    fl, fu = oracle.ibp_bounds(on, l0.astype(np.float64), u0.astype(np.float64))
    lbk, ubk = outward_f32(*(bound * np.concatenate([f[k] for k in range(1, on.n)], axis=1) for f in (fl, fu)))
    rho = (dual * rng.uniform(-1, 1, (B, lbk.shape[1]))).astype(np.float32)
    if zero_rows:
        rho[0] = 0
    return specs, on, l0, u0, lbk, ubk, rho


def _check(got, q, on, l0, u0, lbk, ubk, rho, g):
    far = lambda l, u: np.maximum(np.abs(l.astype(np.float64)), np.abs(u.astype(np.float64)))
    size = np.abs(q) + (np.abs(rho.astype(np.float64)) * far(lbk, ubk)).sum(1) + (np.abs(g[0]) * far(l0, u0)).sum(1)
    for k in range(1, on.n):
        size = size + (np.abs(g[k]) * far(oracle.layer_lists(on, lbk)[k], oracle.layer_lists(on, ubk)[k])).sum(1)
    assert np.all(got <= q + 1e-12 * size)
    assert np.all(q - got <= 1e-11 * size)


CASES = {
    "one": dict(dual=1.0, zero_rows=True),
    "large_sums": dict(dual=1e36),
    "large_terms": dict(dual=1e30, bound=1e12),
    "tiny": dict(dual=1e-25, last=1e-25, zero_rows=True),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("name", sorted(NETS))
def test_as_close_as_fp64_sums(name, case):
    specs, on, l0, u0, lbk, ubk, rho = _problem(name, **CASES[case])
    B = rho.shape[0]
    masks = np.zeros(rho.shape, np.int8)
    net = ldb.Net(specs)
    got = ldb.ld_bound(net, l0, u0, lbk, ubk, np.zeros(B, np.int32), masks, n_iters=0, rho_in=rho,
                       opts=ldb.Options(init="given")).cpu().numpy()
    rep = lambda a: np.repeat(a.astype(np.float64), B, axis=0)
    lo, up, _ = oracle.apply_masks(on, oracle.layer_lists(on, rep(lbk)), oracle.layer_lists(on, rep(ubk)), masks)
    sol = oracle.inner_minimisation(on, rep(l0), rep(u0), lo, up, oracle.layer_lists(on, rho.astype(np.float64)))
    _check(got, sol.q, on, l0, u0, lbk, ubk, rho, sol.g)


@pytest.mark.parametrize("name", sorted(NETS))
def test_ball_norm(name):
    """The l2 ball's term -eps ||g_0|| is as exact as the others: ||g_0||^2 is an FP64 sum, not an error bound."""
    specs, on, l0, u0, lbk, ubk, rho = _problem(name, dual=1.0, zero_rows=True)
    B, eps = rho.shape[0], np.float32(3.0)
    masks = np.zeros(rho.shape, np.int8)
    c = (l0 + u0) / 2
    got = ldb.ld_bound_ball(ldb.Net(specs), c, [eps], lbk, ubk, np.zeros(B, np.int32), masks, n_iters=0, rho_in=rho,
                            opts=ldb.Options(init="given", engine="layerwise")).cpu().numpy()
    rep = lambda a: np.repeat(a.astype(np.float64), B, axis=0)
    lo, up, _ = oracle.apply_masks(on, oracle.layer_lists(on, rep(lbk)), oracle.layer_lists(on, rep(ubk)), masks)
    sol = oracle.inner_minimisation(on, rep(c), rep(c), lo, up, oracle.layer_lists(on, rho.astype(np.float64)),
                                    ball_eps=np.full(B, np.float64(eps)))
    _check(got, sol.q, on, c, c, lbk, ubk, rho, sol.g)
