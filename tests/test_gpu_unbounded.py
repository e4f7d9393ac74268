"""GPU: the final bound where a lower bound is infinite.

Infinite intermediate bounds are valid input (a bound nobody computed).  Without
iterations a blocking ReLU has the dual 0 and contributes 0 whatever its lower
bound is, so the result is bitwise that of any finite lower bound.
"""
import numpy as np
import pytest
import torch

import oracle
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


def _mlp(widths=(12, 64, 33, 1), seed=5):
    specs = synth.make_mlp(list(widths), seed=seed)
    net = oracle_net(specs)
    c = np.random.default_rng(seed).uniform(-1, 1, (1, widths[0])).astype(np.float32)
    l0, u0 = c - np.float32(0.1), c + np.float32(0.1)
    lb, ub = oracle.ibp_bounds(net, l0.astype(np.float64), u0.astype(np.float64))
    lbk, ubk = outward_f32(np.concatenate([lb[k] for k in range(1, net.n)], 1),
                           np.concatenate([ub[k] for k in range(1, net.n)], 1))
    return specs, net, l0, u0, lbk, ubk


@pytest.mark.parametrize("engine", ["layerwise", "fused"])
@pytest.mark.parametrize("init", ["crown", "zero"])
@pytest.mark.parametrize("kind", ["mlp", "conv"])
def test_blocking_neuron_without_a_lower_bound(kind, init, engine):
    if kind == "mlp":
        specs, _, l0, u0, lbk, ubk = _mlp()
    else:
        pb = conv_problem("base", 1)
        specs, l0, u0, lbk, ubk = (pb[k] for k in ("specs", "l0", "u0", "lbk", "ubk"))
    B = 3
    amb = np.nonzero((lbk[0] < 0) & (ubk[0] > 0))[0]
    masks = np.zeros((B, lbk.shape[1]), np.int8)
    masks[1, amb[0]] = masks[2, amb[-1]] = -1
    l0, u0, lbk, ubk = (np.repeat(a, B, 0) for a in (l0, u0, lbk, ubk))
    off = (ubk <= 0) | (masks < 0)
    assert off[1:].any(1).all()
    net = ldb.Net(specs)
    o = ldb.Options(engine=engine, init=init)
    run = lambda end: ldb.ld_bound(net, l0, u0, np.where(off, np.float32(end), lbk), ubk, np.arange(B), masks, n_iters=0,
                                   opts=o).cpu().numpy()
    got = run(-np.inf)
    assert np.isfinite(got).all()
    assert np.array_equal(got, run(-1e3))
