"""GPU: CROWN/WK bounds of convs with one input channel, up to the most weights a layer may have.

The staged weights of a conv are padded to four channels, so a layer of 9216
weights and one channel takes 147 KB of shared memory; first layers (the box
step) and inner layers, against the FP64 oracle with the tolerances of the usual
nets: outward and within 1e-4, FSB's children 1e-4.
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import branching as br
from oracle import intermediate as ib
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import outward_f32

pytestmark = pytest.mark.gpu

NETS = {  # input shape, convs (cout, k, stride, pad), FC widths
    "gray": ((1, 9, 7), [(5, 3, 1, 1), (6, 4, 2, 1)], [11, 1]),
    "gray_1024": ((1, 4, 4), [(1024, 3, 1, 1)], [6, 1]),
    "inner_1024": ((3, 5, 5), [(1, 3, 1, 1), (1024, 3, 2, 0)], [7, 1]),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


@pytest.mark.parametrize("name", sorted(NETS))
def test_crown_wk_and_children(name):
    shape, convs, fcs = NETS[name]
    rng = np.random.default_rng(len(name))
    c0 = rng.uniform(-0.5, 0.5, int(np.prod(shape)))
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
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
                     oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs])
    l0, u0 = (c0 - 0.04).astype(np.float32)[None], (c0 + 0.04).astype(np.float32)[None]
    l64, u64 = l0.astype(np.float64), u0.astype(np.float64)
    flat = lambda lst: np.concatenate([lst[k] for k in range(1, on.n)], axis=1)
    net = ldb.Net(specs)
    gl, gu = (t.cpu().numpy() for t in ldb.ld_intermediate_bounds_propagated(net, l0, u0))
    fl, fu = (flat(f) for f in ib.crown_wk_bounds(on, l64, u64))
    scale = np.maximum(np.abs(fl), np.abs(fu)) + 1.0
    assert np.all(gl <= fl + 1e-12 * scale) and np.all(gu >= fu - 1e-12 * scale)
    assert np.max((fl - gl) / scale) < 1e-4 and np.max((gu - fu) / scale) < 1e-4
    lbk, ubk = outward_f32(*(flat(f) for f in oracle.ibp_bounds(on, l64, u64)))
    _, child = ldb.ld_branch(net, l0, u0, lbk, ubk, B=1, rule="fsb", return_child_bounds=True)
    lo, up = oracle.layer_lists(on, lbk.astype(np.float64)), oracle.layer_lists(on, ubk.astype(np.float64))
    cand = br.fsb_candidates(on, lo, up)
    _, fc = br.fsb_decision(on, l64, u64, lo, up)
    got, fin = child.cpu().numpy(), cand >= 0
    assert np.all(got[fin] <= fc[fin] + 1e-9 * np.maximum(np.abs(fc[fin]), 1.0))
    assert np.max(np.abs(got[fin] - fc[fin]) / np.maximum(np.abs(fc[fin]), 1.0)) < 1e-4
