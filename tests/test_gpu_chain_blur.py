"""Sparse lattices blurred chain by chain: chains of two vertices up to lengths around the rows
loaded together (4), around the longest walked (64) and beyond it (direction lists), and a
dimension whose pass count needs the values rescaled, against the FP64 oracle.

Tolerances as for the other products: 1e-5 relative L2 (fp32 values, ~1e-6 expected), 1e-2 for
bf16 values."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def points_with_run(n, d, length, seed):
    """n scattered points, and `length` points one lattice step along u_0 apart."""
    ls = np.ones(d, np.float32)
    X = 3.0 * synth.gmm_points(n + 1, d, seed)
    E = OracleLattice(np.eye(d, dtype=np.float32), ls).export()["y"].T  # elevation, [D][d]
    u = -np.ones(d + 1)
    u[0] += d + 1
    step = np.linalg.lstsq(E, u, rcond=None)[0]
    run = X[n] + step * (np.arange(length) - length / 2)[:, None]
    return np.ascontiguousarray(np.concatenate([X[:n], run]), np.float32)


def compare(X, k, values, tol):
    n, d = X.shape
    V = synth.gaussian_values(n, k, 9)
    G = synth.gaussian_values(n, k, 10)
    ls = np.ones(d, np.float32)
    ref = OracleLattice(X, ls)
    Xd, lsd = torch.from_numpy(X).cuda(), torch.from_numpy(ls).cuda()
    lat = Lattice(Xd, lsd, spacing=ref.s, value_dtype=values)
    assert lat.m == ref.m and lat.sparse_blur
    for blur, mode in (("sequential", 0), ("transpose", 1), ("symmetric", 2)):
        got = lat.mvm(torch.from_numpy(V).cuda(), blur=blur, alpha=0.7, beta=0.1).cpu().numpy()
        want = ref.mvm(V.astype(np.float64), mode=mode, alpha=0.7, beta=0.1)
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), blur
    if values == "f32":
        grads = lat.mvm_backward(Xd, lsd, torch.from_numpy(V).cuda(), torch.from_numpy(G).cuda(),
                                 blur="symmetric", alpha=0.7)
        exact = ref.mvm_backward(V.astype(np.float64), G.astype(np.float64), mode=2, alpha=0.7)
        for a, b in zip(grads, exact):
            assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-4 * np.linalg.norm(b)


@pytest.mark.parametrize("length", [2, 3, 4, 5, 8, 60, 63, 64, 65, 200])
def test_chain_lengths(length):
    compare(points_with_run(60, 20, length, 3), 5, "f32", 1e-5)


@pytest.mark.parametrize("d,k", [(50, 9), (63, 1), (64, 2), (90, 12), (127, 4)])
@pytest.mark.parametrize("values,tol", [("f32", 1e-5), ("bf16", 1e-2)])
def test_dimensions(d, k, values, tol):
    compare(synth.gmm_points(40, d, 5), k, values, tol)


def test_repeated_points():
    """Few vertices for many entries: the links are read off the neighbour table."""
    X = np.repeat(synth.gmm_points(50, 20, 6), 12, axis=0)
    compare(X, 3, "f32", 1e-5)


def test_wider_stencil_keeps_direction_lists():
    X = synth.gmm_points(200, 30, 7)
    ls = np.ones(30, np.float32)
    V = synth.gaussian_values(200, 3, 9)
    ref = OracleLattice(X, ls, 1, 2)  # RBF, coverage spacing, order 2
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, kernel="rbf_coverage", order=2, spacing=ref.s)
    assert lat.sparse_blur
    got = lat.mvm(torch.from_numpy(V).cuda(), blur="symmetric").cpu().numpy()
    want = ref.mvm(V.astype(np.float64), mode=2)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
