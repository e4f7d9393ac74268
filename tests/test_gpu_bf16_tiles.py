"""GPU: the layer-wise BF16 conv passes at the edges of their tiles.

Planes of 2 to 32 rows (several subdomains a tile, several tiles a subdomain),
batches that leave ragged tiles, odd and even numbers of 8-channel K chunks,
strides and paddings whose phases come in either order, many channels, and
planes without halo tiles (rows no divisor or multiple of 16, columns no
multiple of 8, chunks in descending order).  Short runs against the oracle with
the same operand rounding, with the tolerance of the usual nets' short runs
(1e-5: FP32 sums of exact products); a subdomain's result does not depend on
the rows beside it, NaN duals of a neighbour included.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import outward_f32

pytestmark = pytest.mark.gpu

# name: input shape, convs (cout, k, stride, pad), subdomains
NETS = {
    "odd_chunks": ((3, 16, 16), [(8, 4, 2, 1), (12, 3, 1, 1)], 5),
    "taps_25": ((5, 8, 8), [(8, 3, 1, 1), (7, 5, 1, 2)], 3),
    "flat": ((3, 8, 32), [(16, 4, 2, 1), (24, 4, 2, 1)], 11),
    "several_tiles": ((9, 32, 32), [(20, 3, 1, 1), (33, 4, 2, 1)], 2),
    "channels": ((3, 16, 16), [(32, 4, 2, 1), (33, 3, 1, 1)], 7),
    "rows_24": ((2, 24, 16), [(6, 3, 1, 1)], 3),
    "cols_4": ((3, 8, 8), [(16, 4, 2, 1), (10, 3, 1, 1)], 9),
    "phase_order": ((3, 32, 32), [(8, 3, 2, 1), (8, 2, 2, 0)], 3),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


def _problem(name, props=1):
    shape, convs, B = NETS[name]
    rng = np.random.default_rng(sorted(NETS).index(name) + 70)
    c0 = rng.uniform(-0.5, 0.5, int(np.prod(shape)))
    specs = []
    for cout, k, s, p in convs:
        L = synth.LayerSpec("conv", rng.normal(0, np.sqrt(2 / (shape[0] * k * k)), (cout, shape[0], k, k)).astype(np.float32),
                            rng.normal(0, 0.1, cout).astype(np.float32), shape, s, p)
        specs.append(L)
        shape = L.out_shape
    n = int(np.prod(shape))
    for m in (20, 1):
        specs.append(synth.LayerSpec("fc", rng.normal(0, np.sqrt(2 / n), (m, n)).astype(np.float32),
                                     rng.normal(0, 0.1, m).astype(np.float32), (n,)))
        n = m
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
                     oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs])
    c0 = c0 + rng.uniform(-0.05, 0.05, (props, c0.size)) * (np.arange(props) > 0)[:, None]
    l0, u0 = (c0 - 0.02).astype(np.float32), (c0 + 0.02).astype(np.float32)
    fl, fu = oracle.ibp_bounds(on, l0.astype(np.float64), u0.astype(np.float64))
    flat = [np.concatenate([f[k] for k in range(1, on.n)], axis=1) for f in (fl, fu)]
    lbk, ubk = outward_f32(*flat)
    amb = np.nonzero((lbk[0] < 0) & (ubk[0] > 0))[0]
    masks = synth.split_masks(lbk.shape[1], B, amb, (0, 4), block=3)
    return specs, on, l0, u0, lbk, ubk, (np.arange(B) % props).astype(np.int32), masks


# subdomains of one property, and of several in turn (every tile of columns mixes them)
@pytest.mark.parametrize("name,props", [(n, 1) for n in sorted(NETS)] + [("odd_chunks", 2), ("cols_4", 3)])
def test_short_runs_match_bf16_oracle(name, props):
    specs, on, l0, u0, lbk, ubk, prop, masks = _problem(name, props)
    net = ldb.Net(specs)
    opts = ldb.Options(precision="bf16", engine="layerwise")
    for T in (1, 3):
        out = ldb.ld_bound(net, l0, u0, lbk, ubk, prop, masks, n_iters=T, opts=opts).cpu().numpy()
        ref, _, _ = oracle.ld_bound(on, *(a.astype(np.float64) for a in (l0, u0, lbk, ubk)), prop, masks, T,
                                    operands="bf16")
        fin = np.isfinite(ref)
        assert np.array_equal(np.isfinite(out), fin)
        assert np.max(np.abs(out[fin] - ref[fin]) / np.maximum(np.abs(ref[fin]), 1.0)) < 1e-5


@pytest.mark.parametrize("name", sorted(NETS))
def test_rows_are_independent(name):
    specs, on, l0, u0, lbk, ubk, prop, masks = _problem(name)
    net = ldb.Net(specs)
    opts = ldb.Options(precision="bf16", engine="layerwise", init="given")
    rho = (0.1 * np.random.default_rng(1).normal(size=masks.shape)).astype(np.float32)
    run = lambda r: ldb.ld_bound(net, l0, u0, lbk, ubk, prop[: len(r)], masks[: len(r)], n_iters=2, opts=opts,
                                 rho_in=torch.from_numpy(r).cuda(), return_rho=True)[1].cpu().numpy()
    whole = run(rho)
    assert np.isfinite(whole).all()
    bad = rho.copy()
    bad[1] = np.nan
    got = run(bad)
    keep = np.arange(len(rho)) != 1
    assert np.array_equal(got[keep], whole[keep])
