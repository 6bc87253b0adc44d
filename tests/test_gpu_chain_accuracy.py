"""Sparse fp32 products carry no common factor: the blur leaves a power of the centre tap to the
slice, which must not put that power's fp32 rounding error (up to 6e-8) on every value alike.

The factor is read off as <got, exact> / <exact, exact>.  Rounding errors of single values (1e-7
relative, random) move it by about 1e-7 / sqrt(16,000 values) = 8e-10; the bound is 1e-8."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("d", [14, 20, 25, 50, 90])
def test_common_factor(d):
    n, k = 2000, 8
    X = synth.gmm_points(n, d, 2)
    ls = np.ones(d, np.float32)
    V, G = synth.gaussian_values(n, k, 11), synth.gaussian_values(n, k, 12)
    ref = OracleLattice(X, ls)
    lat = Lattice(gpu(X), gpu(ls), spacing=ref.s)
    assert lat.sparse_blur

    def factor(got, want):
        return float((got.cpu().numpy().astype(np.float64) * want).sum() / (want * want).sum())

    want = ref.mvm(V.astype(np.float64), mode=2)
    out = lat.mvm(gpu(V), blur="symmetric")
    dV, _, _ = lat.mvm_backward(gpu(X), gpu(ls), gpu(V), gpu(G), blur="symmetric")
    f = factor(out, want), factor(dV, ref.mvm(G.astype(np.float64), mode=2))
    print("d=%d: product 1 %+.1e, dV 1 %+.1e" % (d, f[0] - 1, f[1] - 1))
    assert max(abs(x - 1) for x in f) <= 1e-8


@pytest.mark.parametrize("d", [14, 20, 90])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinities_stay(d, value):
    """An entry that is not finite reaches the points that share vertices with it, as it is (all
    taps and weights are positive); the others keep their bits."""
    n = 300
    X = synth.gmm_points(n, d, 7)
    ref = OracleLattice(X, np.ones(d, np.float32))
    lat = Lattice(gpu(X), 1.0, spacing=ref.s)
    assert lat.sparse_blur
    one = np.zeros((n, 1))
    one[n // 2] = 1.0
    V = synth.gaussian_values(n, 1, 3)
    W = V.copy()
    W[n // 2] = value
    for blur, mode in (("symmetric", 2), ("sequential", 0)):
        got = lat.mvm(gpu(W), blur=blur).cpu().numpy()
        other = lat.mvm(gpu(V), blur=blur).cpu().numpy()
        hit = ref.mvm(one, mode=mode) != 0.0
        assert np.array_equal(got[~hit], other[~hit])
        assert hit[n // 2] and np.array_equal(got[hit], np.full(hit.sum(), value, np.float32),
                                              equal_nan=True)
