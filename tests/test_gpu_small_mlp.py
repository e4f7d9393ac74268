"""GPU: the shared-memory form of the fused iterations for small FC nets.

It has to be bitwise the general fused kernel, whose l2-ball form still runs on
such nets: over balls of radius zero the input set is the point c, as over the
box [c, c], so the two forms see one problem.  Widths around the edges of the
vector and split paths (a multiple of 4 or not, one or several 16-row batches,
more columns and rows than the CTA has threads and warps), every launch shape,
(except where the ball form itself runs layer-wise: it needs a float of FC
scratch per warp), ragged batches, an empty subdomain, a launch longer than one step table, and a
run resumed from its duals and moments.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth
from helpers import oracle_net, outward_f32

pytestmark = pytest.mark.gpu

WIDTHS = [[10, 20, 20, 1], [7, 5, 1], [12, 64, 33, 18, 1], [40, 100, 16, 1], [300, 24, 100, 1]]
SHAPES = [(1, 512), (2, 512), (1, 256), (2, 256), (4, 256)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


def _problem(widths, radius=0.0, B=9):
    specs = synth.make_mlp(widths, seed=sum(widths))
    net = oracle_net(specs)
    rng = np.random.default_rng(widths[0])
    c = rng.uniform(-1, 1, (1, widths[0])).astype(np.float32)
    l0, u0 = (c - np.float32(radius)), (c + np.float32(radius))
    wide = 0.1      # intermediate bounds of a larger box: valid, and ambiguous ReLUs to choose at
    lb, ub = oracle.ibp_bounds(net, c.astype(np.float64) - wide, c.astype(np.float64) + wide)
    lbk, ubk = outward_f32(np.concatenate([lb[k] for k in range(1, net.n)], 1),
                           np.concatenate([ub[k] for k in range(1, net.n)], 1))
    amb = np.nonzero((lbk[0] < 0) & (ubk[0] > 0))[0]
    masks = synth.split_masks(lbk.shape[1], B, amb, (0, 3), block=3)
    return specs, net, c, l0, u0, lbk, ubk, masks


@pytest.mark.parametrize("tile,threads", SHAPES)
@pytest.mark.parametrize("widths", WIDTHS, ids=lambda w: "-".join(map(str, w)))
def test_bitwise_the_general_kernel(widths, tile, threads):
    if sum((max(w, 2 * i if i % 4 == 0 and i // 2 <= threads else 0) + 3) // 4 * 4
           for i, w in zip(widths[:-2], widths[1:-1])) < threads // 32:
        pytest.skip("the ball form has no FC scratch for its norm here and runs layer-wise")
    specs, _, c, l0, u0, lbk, ubk, masks = _problem(widths)
    net = ldb.Net(specs)
    o = ldb.Options(engine="fused", tile=tile, cta_threads=threads)
    box = ldb.ld_bound(net, l0, u0, lbk, ubk, None, masks, n_iters=13, opts=o, return_rho=True)
    ball = ldb.ld_bound_ball(net, c, [0.0], lbk, ubk, None, masks, n_iters=13, opts=o, return_rho=True)
    assert torch.equal(box[1], ball[1])


def test_against_the_oracle_and_resumed():
    specs, on, c, l0, u0, lbk, ubk, masks = _problem([40, 100, 16, 1], radius=0.1, B=5)
    masks[3] = 0
    lbe, ube = np.repeat(lbk, 2, 0), np.repeat(ubk, 2, 0)
    lbe[1, 0], ube[1, 0] = 1.0, -1.0          # property 1: an empty ReLU interval
    prop = np.array([0, 0, 0, 1, 0], np.int32)
    net = ldb.Net(specs)
    o = ldb.Options(engine="fused", tile=1, cta_threads=512)
    two = lambda a: np.repeat(a, 2, 0)
    out, rho = ldb.ld_bound(net, two(l0), two(u0), lbe, ube, prop, masks, n_iters=3, opts=o, return_rho=True)
    f = lambda a: a.astype(np.float64)
    ref, _, _ = oracle.ld_bound(on, f(l0), f(u0), f(lbk), f(ubk), None, masks, 3)
    got = out.cpu().numpy()
    assert np.isposinf(got[3])
    keep = [0, 1, 2, 4]
    assert np.max(np.abs(got[keep] - ref[keep]) / np.maximum(np.abs(ref[keep]), 1.0)) < 1e-5
    # 140 iterations (two step tables) in one call and as 100 + 40
    mv = torch.zeros((2, 5, net.N), device="cuda")
    run = lambda T, **k: ldb.ld_bound(net, l0, u0, lbk, ubk, None, masks, n_iters=T, return_rho=True, **k)
    whole = run(140, opts=o)
    p = ldb.Options(**{**o.__dict__, "t_total": 140})
    first = run(100, opts=p, adam_mv=mv)
    q = ldb.Options(**{**p.__dict__, "t_offset": 100, "init": "given"})
    second = run(40, opts=q, rho_in=first[1], adam_mv=mv)
    assert torch.equal(whole[1], second[1]) and torch.equal(whole[0], second[0])
