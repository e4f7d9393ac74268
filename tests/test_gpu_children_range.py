"""GPU: FSB's children bounds (FP64) where a row's scalar terms leave FP32's middle range.

One hidden layer with one ambiguous ReLU (bounds -1 to 1), so that both of its
children's bounds are known; the other ReLUs pass.  The products of bias and
coefficient and of box and coefficient are larger than any FP32 number, of
ordinary size, or below 2^-102, where an FP32 product has no exact low part.
Sound, and within 1e-6 of the FP64 oracle (an FP32 coefficient's rounding, 2^-24,
times a margin for cancellation).
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import branching as br
from paper_2104_06718_gb300 import binding as ldb
from paper_2104_06718_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    build.build()
    ldb.load_library()


@pytest.mark.parametrize("scale", [(1e15, 1e12, 1e15), (1.0, 1.0, 1.0), (1e-13, 1e-12, 1e-8)],
                         ids=["large", "one", "tiny"])
def test_children(scale):
    s1, s2, sx = scale
    rng = np.random.default_rng(8)
    n0, h = 40, 21
    W1 = (s1 * rng.uniform(0.5, 1.0, (h, n0)) * np.where(rng.random((h, n0)) < 0.5, -1, 1)).astype(np.float32)
    b1 = (s1 * sx * rng.uniform(60, 80, h)).astype(np.float32)
    b1[4] = 0
    W2 = (s2 * rng.uniform(-1.0, 1.0, (1, h))).astype(np.float32)
    specs = [synth.LayerSpec("fc", W1, b1, (n0,)), synth.LayerSpec("fc", W2, np.zeros(1, np.float32), (h,))]
    on = oracle.Net([oracle.Layer("fc", s.W, s.b) for s in specs])
    l0 = (sx * rng.uniform(-1.0, 0.9, (1, n0))).astype(np.float32)
    u0 = (l0 + np.float32(0.1 * sx)).astype(np.float32)
    lbk, ubk = (b1 - np.float32(50 * s1 * sx))[None], (b1 + np.float32(50 * s1 * sx))[None]
    unit = 1.0 if s1 >= 1 else s1 * sx
    lbk[0, 4], ubk[0, 4] = -unit, unit
    assert (lbk[0, np.arange(h) != 4] > 0).all() and np.isfinite(ubk).all()
    _, child = ldb.ld_branch(ldb.Net(specs), l0, u0, lbk, ubk, B=1, rule="fsb", return_child_bounds=True)
    f = lambda a: a.astype(np.float64)
    got = child.cpu().numpy()[0]
    for half, phase in enumerate((+1, -1)):
        lo, up = br.split_bounds(on, oracle.layer_lists(on, f(lbk)), oracle.layer_lists(on, f(ubk)), [4], [phase])
        ref = br.output_bound_best(on, f(l0), f(u0), lo, up)[0]
        assert np.all(got[:, half] <= ref)
        assert np.all(ref - got[:, half] <= 1e-6 * abs(ref))
