"""GPU: the FP64 final bound at given duals, at the edges of its blocks and levels.

FC sums of 1, 63, 64, 65 and 129 terms (blocks of 64), convs of odd channel
counts with and without a blocked path, duals that are zero, of one size, or
spread over 18 decades (the levels' exponents follow the largest products).
Sound: at most the FP64 oracle's q at the same duals (its own rounding, 1e-12 of
the terms' size, allowed for); close: within 1e-9 of it at duals of one size
(the tolerance of the usual nets), 1e-9 of the terms' size at spread ones.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import outward_f32

pytestmark = pytest.mark.gpu

# name: input shape, convs (cout, k, stride, pad), FC widths (the last 1)
NETS = {
    "fc_edges": ((129,), [], [64, 65, 63, 1, 1]),
    "fc_wide": ((7,), [], [200, 130, 1]),
    "conv_k4": ((3, 12, 12), [(6, 4, 2, 1), (8, 4, 2, 1)], [65, 1]),
    "conv_k3": ((5, 7, 9), [(9, 3, 1, 1), (4, 3, 1, 0)], [33, 1]),
    "conv_k5": ((2, 9, 9), [(7, 5, 2, 2)], [64, 1]),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


@pytest.mark.parametrize("duals", ["zero", "even", "spread"])
@pytest.mark.parametrize("name", sorted(NETS))
def test_sound_and_close(name, duals):
    shape, convs, fcs = NETS[name]
    rng = np.random.default_rng(sorted(NETS).index(name) + 90)
    c0 = rng.uniform(-0.5, 0.5, int(np.prod(shape)))
    specs = []
    for cout, k, s, p in convs:
        specs.append(synth.LayerSpec(
            "conv", rng.normal(0, np.sqrt(2 / (shape[0] * k * k)), (cout, shape[0], k, k)).astype(np.float32),
            rng.normal(0, 0.1, cout).astype(np.float32), shape, s, p))
        shape = specs[-1].out_shape
    n = int(np.prod(shape))
    for m in fcs:
        specs.append(synth.LayerSpec("fc", rng.normal(0, np.sqrt(2 / n), (m, n)).astype(np.float32),
                                     rng.normal(0, 0.1, m).astype(np.float32), (n,)))
        n = m
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
                     oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs])
    l0, u0 = (c0 - 0.05).astype(np.float32)[None], (c0 + 0.05).astype(np.float32)[None]
    fl, fu = oracle.ibp_bounds(on, l0.astype(np.float64), u0.astype(np.float64))
    lbk, ubk = outward_f32(*(np.concatenate([f[k] for k in range(1, on.n)], axis=1) for f in (fl, fu)))
    B = 5
    masks = np.zeros((B, lbk.shape[1]), np.int8)
    rho = rng.normal(0, 0.3, masks.shape)
    if duals == "zero":
        rho *= 0
    if duals == "spread":
        rho *= 10.0 ** rng.uniform(-12, 6, rho.shape)
    rho = rho.astype(np.float32)
    out = ldb.ld_bound(ldb.Net(specs), l0, u0, lbk, ubk, np.zeros(B, np.int32), masks, n_iters=0, rho_in=rho,
                       opts=ldb.Options(init="given")).cpu().numpy()
    rep = lambda a: np.repeat(a.astype(np.float64), B, axis=0)
    lo, up, _ = oracle.apply_masks(on, oracle.layer_lists(on, rep(lbk)), oracle.layer_lists(on, rep(ubk)), masks)
    q = oracle.inner_minimisation(on, rep(l0), rep(u0), lo, up, oracle.layer_lists(on, rho.astype(np.float64))).q
    size = np.maximum(np.abs(q), 1.0)
    if duals == "spread":
        size = size + (np.abs(rho.astype(np.float64)) * np.maximum(np.abs(lbk), np.abs(ubk))).sum(1)
    assert np.all(out <= q + 1e-12 * size)
    assert np.all(q - out <= 1e-9 * size)
