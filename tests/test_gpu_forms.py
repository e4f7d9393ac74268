"""GPU: forms of the kernels that the nets of the other tests do not reach.

  * Nets of one hidden layer run on the shared-memory kernel or the general fused
    kernel by batch size: the same subdomains in a small and a large batch, on a real
    box, bitwise (the input layer's columns, their row order and halves are in it),
    and the shared-memory kernel against the FP64 oracle on real boxes (1e-5, as for
    the usual nets after three iterations).
  * CROWN/WK bounds where a conv follows an FC layer, and FC layers at the edges of
    their units of two and eight inputs, rounds of eight and staged 128 rows: outward
    and within 1e-4 of the oracle, a row the same alone and in a batch.
  * BF16 layer-wise passes with and without the state's prefetch (by batch size): the
    same subdomains, bitwise.
  * DSG+ before and after a proximal call that grows the workspace of both.
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import intermediate as ib
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import conv_problem, oracle_net, outward_f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


def _mlp(widths, radius=0.1):
    specs = synth.make_mlp(widths, seed=sum(widths))
    on = oracle_net(specs)
    c = np.random.default_rng(widths[0]).uniform(-1, 1, (1, widths[0])).astype(np.float32)
    l0, u0 = c - np.float32(radius), c + np.float32(radius)
    lb, ub = oracle.ibp_bounds(on, l0.astype(np.float64), u0.astype(np.float64))
    lbk, ubk = outward_f32(np.concatenate([lb[k] for k in range(1, on.n)], 1),
                           np.concatenate([ub[k] for k in range(1, on.n)], 1))
    amb = np.nonzero((lbk[0] < 0) & (ubk[0] > 0))[0]
    return specs, on, l0, u0, lbk, ubk, amb


@pytest.mark.parametrize("widths,tile,threads,large", [
    ([300, 24, 1], 2, 256, 2000), ([300, 24, 1], 4, 256, 2001), ([302, 40, 1], 2, 256, 1500),
    ([784, 24, 1], 1, 512, 200), ([700, 24, 1], 1, 512, 400)])
def test_one_hidden_layer_in_small_and_large_batches(widths, tile, threads, large):
    specs, _, l0, u0, lbk, ubk, amb = _mlp(widths)
    masks = np.zeros((large, lbk.shape[1]), np.int8)
    masks[:9] = synth.split_masks(lbk.shape[1], 9, amb, (0, 3), block=3)
    net = ldb.Net(specs)
    o = ldb.Options(engine="fused", tile=tile, cta_threads=threads)
    run = lambda n: ldb.ld_bound(net, l0, u0, lbk, ubk, None, masks[:n], n_iters=13, opts=o, return_rho=True)
    (a, ra), (b, rb) = run(9), run(large)
    assert torch.equal(ra, rb[:9]) and torch.equal(a, b[:9])


@pytest.mark.parametrize("tile,threads", [(1, 512), (2, 256), (4, 256)])
@pytest.mark.parametrize("widths", [[10, 20, 20, 1], [7, 5, 1], [12, 64, 33, 18, 1], [300, 24, 100, 1], [257, 9, 1]],
                         ids=lambda w: "-".join(map(str, w)))
def test_shared_memory_kernel_on_boxes(widths, tile, threads):
    specs, on, l0, u0, lbk, ubk, amb = _mlp(widths)
    masks = synth.split_masks(lbk.shape[1], 7, amb, (0, 2), block=5)
    f = lambda a: a.astype(np.float64)
    got = ldb.ld_bound(ldb.Net(specs), l0, u0, lbk, ubk, None, masks, n_iters=3,
                       opts=ldb.Options(engine="fused", tile=tile, cta_threads=threads)).cpu().numpy()
    ref, _, _ = oracle.ld_bound(on, f(l0), f(u0), f(lbk), f(ubk), None, masks, 3)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    assert np.max(np.abs(got[fin] - ref[fin]) / np.maximum(np.abs(ref[fin]), 1.0)) < 1e-5


# layers: an int (FC width) or (in_shape, cout, k, stride, pad)
IB_NETS = {
    "conv_after_fc": (11, [48, ((3, 4, 4), 6, 3, 1, 1), ((6, 4, 4), 5, 4, 2, 1), 9, 1]),
    "units": (17, [9, 129, 8, 3, 1]),
    "ones": (1, [1, 2, 1, 1]),
    "edges_1023": (1023, [5, 16, 1]),
    "edges_1025": (1025, [15, 7, 1]),
}


@pytest.mark.parametrize("name", sorted(IB_NETS))
def test_crown_wk_forms(name):
    n, layers = IB_NETS[name]
    rng = np.random.default_rng(len(name) + 3)
    c = rng.uniform(-0.5, 0.5, n)
    specs = []
    for d in layers:
        if isinstance(d, int):
            specs.append(synth.LayerSpec("fc", rng.normal(0, np.sqrt(2 / n), (d, n)).astype(np.float32),
                                         rng.normal(0, 0.1, d).astype(np.float32), (n,)))
            n = d
        else:
            shape, cout, k, s, p = d
            W = rng.normal(0, np.sqrt(2 / (shape[0] * k * k)), (cout, shape[0], k, k)).astype(np.float32)
            specs.append(synth.LayerSpec("conv", W, rng.normal(0, 0.1, cout).astype(np.float32), shape, s, p))
            n = int(np.prod(specs[-1].out_shape))
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) if s.kind == "fc" else
                     oracle.Layer("conv", s.W, s.b, in_shape=s.in_shape, stride=s.stride, pad=s.pad) for s in specs])
    l0, u0 = (c - 0.04).astype(np.float32)[None], (c + 0.04).astype(np.float32)[None]
    net = ldb.Net(specs)
    gl, gu = ldb.ld_intermediate_bounds_propagated(net, l0, u0)
    flat = lambda lst: np.concatenate([lst[k] for k in range(1, on.n)], axis=1)
    fl, fu = (flat(f) for f in ib.crown_wk_bounds(on, l0.astype(np.float64), u0.astype(np.float64)))
    a, b = gl.cpu().numpy(), gu.cpu().numpy()
    scale = np.maximum(np.abs(fl), np.abs(fu)) + 1.0
    assert np.all(a <= fl + 1e-12 * scale) and np.all(b >= fu - 1e-12 * scale)
    assert np.max((fl - a) / scale) < 1e-4 and np.max((b - fu) / scale) < 1e-4
    many = ldb.ld_intermediate_bounds_propagated(net, l0, u0, masks=np.zeros((13, net.N), np.int8))
    assert torch.equal(many[0], gl.expand(13, -1)) and torch.equal(many[1], gu.expand(13, -1))


def test_bf16_passes_in_small_and_large_batches():
    pb = conv_problem("base", 12, block=2)
    net = ldb.Net(pb["specs"])
    large = 1700                             # 108 MB of state
    masks = np.zeros((large, pb["masks"].shape[1]), np.int8)
    masks[:12] = pb["masks"]
    o = ldb.Options(engine="layerwise", precision="bf16")
    run = lambda n: ldb.ld_bound(net, pb["l0"], pb["u0"], pb["lbk"], pb["ubk"], None, masks[:n], n_iters=4, opts=o,
                                 return_rho=True)
    (a, ra), (b, rb) = run(12), run(large)
    assert torch.equal(ra, rb[:12]) and torch.equal(a, b[:12])


def test_dsg_after_a_growing_proximal_call():
    pb = conv_problem("base", 6, block=4)
    net = ldb.Net(pb["specs"])
    a = (net, pb["l0"], pb["u0"], pb["lbk"], pb["ubk"])
    first = ldb.ld_bound_dsg(*a, None, pb["masks"], n_iters=5)
    ldb.ld_bound_proximal(*a, None, np.zeros((64, pb["masks"].shape[1]), np.int8), n_iters=2)
    again = ldb.ld_bound_dsg(*a, None, pb["masks"], n_iters=5)
    assert torch.equal(first[0], again[0])
