"""GPU: the staged and grouped kernels at the edges of their tiles.

Nets whose channel counts, planes, strides, padding and FC widths are not the
usual ones (channels that are no multiple of the blocking, a plane smaller than
a tile, unpadded 3x3, a 5x5 conv and a 2x2 stride-2 conv on the general paths,
FC widths past one staged round, FC layers below FC layers), batches that leave
ragged tiles.  Interval bounds, CROWN/WK bounds (root and per subdomain), the
dual value, supergradient and upper bound at given duals, FSB's children and the
proximal solver's first iteration, each against the FP64 oracle with the
tolerances of the tests of the usual nets: interval and CROWN/WK bounds outward
and within 1e-4, q and the children 1e-5, the proximal bound 1e-5 (twice: the
blocks of one iteration pass their rounding on once).
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import branching as br
from oracle import intermediate as ib
from oracle import proximal as px
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import outward_f32

pytestmark = pytest.mark.gpu

# name: input shape, convs (cout, k, stride, pad), FC widths (the last 1), subdomains
NETS = {
    "channels": ((3, 12, 12), [(6, 4, 2, 1), (5, 3, 1, 1)], [33, 1], 5),
    "unpadded": ((4, 10, 10), [(10, 3, 1, 0), (4, 4, 2, 1)], [17, 1], 7),
    "general": ((2, 11, 9), [(7, 5, 1, 2), (9, 2, 2, 0)], [130, 1], 3),
    "small": ((3, 4, 4), [(4, 4, 2, 1), (12, 3, 1, 1)], [9, 5, 1], 33),
    "wide_in": ((17, 6, 6), [(8, 4, 2, 1)], [150, 70, 1], 6),
    "fc": ((23,), [], [140, 37, 11, 1], 9),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


def _net(name):
    shape, convs, fcs, B = NETS[name]
    rng = np.random.default_rng(sorted(NETS).index(name) + 40)
    l0c = rng.uniform(-0.5, 0.5, int(np.prod(shape)))
    specs = []
    for cout, k, s, p in convs:
        fan = shape[0] * k * k
        L = synth.LayerSpec("conv", rng.normal(0, np.sqrt(2 / fan), (cout, shape[0], k, k)).astype(np.float32),
                            rng.normal(0, 0.1, cout).astype(np.float32), shape, s, p)
        specs.append(L)
        shape = L.out_shape
    n = int(np.prod(shape))
    for m in fcs:
        specs.append(synth.LayerSpec("fc", rng.normal(0, np.sqrt(2 / n), (m, n)).astype(np.float32),
                                     rng.normal(0, 0.1, m).astype(np.float32), (n,)))
        n = m
    layers = [oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
              oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs]
    on = oracle.Net(layers)
    l0 = (l0c - 0.04).astype(np.float32)[None]
    u0 = (l0c + 0.04).astype(np.float32)[None]
    return specs, on, l0, u0, B


def _flat(on, lst):
    return np.concatenate([lst[k] for k in range(1, on.n)], axis=1)


def _outward(gl, gu, fl, fu):
    scale = np.maximum(np.abs(fl), np.abs(fu)) + 1.0
    assert np.all(gl <= fl + 1e-12 * scale) and np.all(gu >= fu - 1e-12 * scale)
    assert np.max((fl - gl) / scale) < 1e-4 and np.max((gu - fu) / scale) < 1e-4


def _problem(name):
    specs, on, l0, u0, B = _net(name)
    fl, fu = oracle.ibp_bounds(on, l0.astype(np.float64), u0.astype(np.float64))
    lbk, ubk = outward_f32(_flat(on, fl), _flat(on, fu))
    amb = np.nonzero((lbk[0] < 0) & (ubk[0] > 0))[0]
    masks = synth.split_masks(lbk.shape[1], B, amb, (0, 3), block=7)
    f64 = lambda a: np.repeat(a.astype(np.float64), B, axis=0)
    lo, up, empty = oracle.apply_masks(on, oracle.layer_lists(on, f64(lbk)), oracle.layer_lists(on, f64(ubk)), masks)
    assert not empty.any()
    return specs, on, l0, u0, lbk, ubk, masks, f64(l0), f64(u0), lo, up


def _close(a, b, tol):
    assert np.max(np.abs(a - b) / np.maximum(np.abs(b), 1.0)) < tol


@pytest.mark.parametrize("name", sorted(NETS))
def test_interval_and_propagated_bounds(name):
    specs, on, l0, u0, lbk, ubk, masks, *_ = _problem(name)
    net = ldb.Net(specs)
    l64, u64 = l0.astype(np.float64), u0.astype(np.float64)
    gl, gu, out = ldb.ld_intermediate_bounds(net, l0, u0, want_output_lb=True)
    fl, fu = oracle.ibp_bounds(on, l64, u64)
    _outward(gl.cpu().numpy(), gu.cpu().numpy(), _flat(on, fl), _flat(on, fu))
    assert out.item() <= fl[on.n][0, 0] + 1e-12 and abs(out.item() - fl[on.n][0, 0]) < 1e-4 * max(1, abs(out.item()))
    gl, gu = ldb.ld_intermediate_bounds_propagated(net, l0, u0)
    fl, fu = ib.crown_wk_bounds(on, l64, u64)
    _outward(gl.cpu().numpy(), gu.cpu().numpy(), _flat(on, fl), _flat(on, fu))
    root = gl
    gl, gu = ldb.ld_intermediate_bounds_propagated(net, l0, u0, masks=masks)
    fl, fu, empty = ib.crown_wk_bounds_split(on, l64, u64, masks)
    ok = ~empty
    _outward(gl.cpu().numpy()[ok], gu.cpu().numpy()[ok], _flat(on, fl)[ok], _flat(on, fu)[ok])
    # a row's bounds do not depend on the rows beside it
    assert torch.equal(gl[0], root[0])
    one, _ = ldb.ld_intermediate_bounds_propagated(net, l0, u0, masks=masks[1:2])
    assert torch.equal(gl[1], one[0])


@pytest.mark.parametrize("name", sorted(NETS))
def test_evaluation_and_children(name):
    specs, on, l0, u0, lbk, ubk, masks, L0, U0, lo, up = _problem(name)
    net = ldb.Net(specs)
    rng = np.random.default_rng(3)
    rho = (0.3 * rng.normal(size=masks.shape)).astype(np.float32)
    q, sg, _ = ldb.ld_dual_supergradient(net, l0, u0, lbk, ubk, rho, masks=masks)
    sol = oracle.inner_minimisation(on, L0, U0, lo, up, oracle.layer_lists(on, rho.astype(np.float64)))
    _close(q.cpu().numpy(), sol.q, 1e-5)
    ref = _flat(on, oracle.supergradient(sol))
    bad = np.abs(sg.cpu().numpy() - ref) > 1e-5 * np.maximum(np.abs(ref), 1.0)
    assert bad.mean() < 2e-3          # near-ties alone
    ub, x0 = ldb.ld_upper_bound(net, l0, u0, lbk, ubk, rho, masks=masks, return_x0=True)
    _close(ub.cpu().numpy(), on.evaluate(x0.cpu().numpy().astype(np.float64)), 1e-5)
    dec, child = ldb.ld_branch(net, l0, u0, lbk, ubk, masks=masks, rule="fsb", return_child_bounds=True)
    cand = br.fsb_candidates(on, lo, up)
    _, fc = br.fsb_decision(on, L0, U0, lo, up)
    got, fin = child.cpu().numpy(), cand >= 0
    assert np.all(got[fin] <= fc[fin] + 1e-9 * np.maximum(np.abs(fc[fin]), 1.0))
    _close(got[fin], fc[fin], 1e-4)


@pytest.mark.parametrize("name", sorted(NETS))
def test_proximal_first_iteration(name):
    specs, on, l0, u0, lbk, ubk, masks, L0, U0, lo, up = _problem(name)
    net = ldb.Net(specs)
    out = ldb.ld_bound_proximal(net, l0, u0, lbk, ubk, masks=masks, n_iters=1).cpu().numpy()
    ref = px.proximal_solver(on, L0, U0, lo, up, 1)
    _close(out, ref.q_final, 2e-5)
    again = ldb.ld_bound_proximal(net, l0, u0, lbk, ubk, masks=masks, n_iters=1).cpu().numpy()
    assert np.array_equal(out, again)
