"""Lattices whose sorts and scans sit at the edges of their kernels: one and two tiles of 4096
items, and 128 tiles, up to which the sort adds up its histograms itself, against the FP64 oracle.

Tolerance as for the other products: 1e-5 relative L2 (fp32 values, ~1e-6 expected)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [
    (2, 3), (3, 1), (2047, 1), (2048, 1), (2049, 1), (4095, 2), (4096, 3), (4097, 2),
    (131072, 3), (131073, 3), (262143, 1), (262145, 1),
])
def test_product_at_sort_edges(n, d):
    X = synth.gmm_points(n, d, 31)
    V = synth.gaussian_values(n, 2, 32)
    ls = np.full(d, 0.25, np.float32)
    ref = OracleLattice(X, ls)
    lat = Lattice(torch.from_numpy(X).cuda(), torch.from_numpy(ls).cuda(), spacing=ref.s)
    assert lat.m == ref.m
    got = lat.mvm(torch.from_numpy(V).cuda(), blur="symmetric").cpu().numpy()
    want = ref.mvm(V.astype(np.float64), mode=2)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
