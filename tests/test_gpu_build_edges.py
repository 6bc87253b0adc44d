"""Lattice construction at the edges of its kernels' ranges, bit-exact against the oracle:
dimensions around the unrolled sizes, point counts around a block of 128, repeated points,
ties, zeros of both signs and lengthscales over many orders of magnitude."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def check(X, ls, **kw):
    ref = OracleLattice(X, ls)
    lat = Lattice(torch.from_numpy(X).cuda(), torch.from_numpy(ls).cuda(), spacing=ref.s, **kw)
    assert lat.m == ref.m
    got, want = lat.export(), ref.export()
    assert np.array_equal(got["keys"][got["idx"]], want["keys"][want["idx"]])
    assert np.array_equal(got["w"], want["w"].astype(np.float32))
    # the blur's neighbours: one product in each order of the directions
    V = synth.gaussian_values(X.shape[0], 3, 5)
    for blur, mode in (("sequential", 0), ("symmetric", 2)):
        out = lat.mvm(torch.from_numpy(V).cuda(), blur=blur).cpu().numpy()
        exact = ref.mvm(V.astype(np.float64), mode=mode)
        assert np.linalg.norm(out - exact) <= 1e-5 * np.linalg.norm(exact)


@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 8, 11, 12, 15, 16, 31, 32, 63, 64])
@pytest.mark.parametrize("n", [1, 127, 128, 385])
def test_dimensions_and_counts(n, d):
    check(synth.gmm_points(max(n, 2), d, 3)[:n], np.ones(d, np.float32))


@pytest.mark.parametrize("d", [2, 5, 20])
def test_ties_zeros_and_repeats(d):
    rng = np.random.default_rng(4)
    X = rng.integers(-2, 3, (300, d)).astype(np.float32)
    X[X == 0] = np.where(rng.random((X == 0).sum()) < 0.5, np.float32(-0.0), np.float32(0.0))
    X[100:200] = X[:100]
    check(X, np.full(d, 0.5, np.float32))


def test_lengthscales_over_many_orders():
    X = synth.gmm_points(257, 6, 8)
    ls = np.float32([1e-2, 1.0, 1e3, 3e38, 1e-38, 7.0])
    X[:, 4] *= 1e-37
    X[:, 3] = 0.0
    check(X, ls)
