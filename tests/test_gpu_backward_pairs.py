"""The symmetric backward's two blurs done as the halves of wider rows: column counts with and
without padding, dense lattices (cluster, launch per pass, too large to be paired), sparse ones,
and gradients asked for one by one, against the FP64 oracle.

Tolerances as for the other lattice gradients: dV 1e-5, dX and dls 1e-4 relative L2."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,d,k", [
    (500, 3, 1), (500, 3, 2), (700, 5, 3), (700, 5, 9), (3000, 9, 1), (6000, 8, 8), (9000, 9, 130),
    (30000, 9, 16), (400, 20, 1), (400, 20, 3), (900, 33, 8), (300, 50, 127), (300, 70, 129),
])
def test_symmetric_gradients(n, d, k):
    X, ls = synth.correlated_points(n, d, 17)
    V = synth.gaussian_values(n, k, 18)
    G = synth.gaussian_values(n, k, 19)
    lat = Lattice(gpu(X), gpu(ls))
    dV, dX, dls = lat.mvm_backward(gpu(X), gpu(ls), gpu(V), gpu(G), blur="symmetric", alpha=0.9)
    rdV, rdX, rdls = OracleLattice(X, ls).mvm_backward(V.astype(np.float64), G.astype(np.float64),
                                                       mode=2, alpha=0.9)
    e = (rel(dV, rdV), rel(dX, rdX), rel(dls, rdls))
    print("n=%d d=%d k=%d m=%d: dV %.1e dX %.1e dls %.1e" % ((n, d, k, lat.m) + e))
    assert e[0] <= 1e-5 and e[1] <= 1e-4 and e[2] <= 1e-4
