"""Sparse lattices with a chain longer than one thread group walks: the build gives the chains up
after 64 steps and lists the vertices by direction.  Runs around the limit and across the whole
key range, along two directions at once, against the FP64 oracle (1e-5 relative L2, ~1e-6
expected), and the time of such a build."""

import time

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def points_with_runs(n, d, lengths, seed):
    """n scattered points, and for each direction j in `lengths` that many points one lattice step
    along u_j apart, centred on the origin."""
    E = OracleLattice(np.eye(d, dtype=np.float32), np.ones(d, np.float32)).export()["y"].T
    X = [3.0 * synth.gmm_points(n, d, seed)]
    for j, length in lengths.items():
        u = -np.ones(d + 1)
        u[j] += d + 1
        step = np.linalg.lstsq(E, u, rcond=None)[0]
        X.append(0.01 + step * (np.arange(length) - length / 2)[:, None])
    return np.ascontiguousarray(np.concatenate(X), np.float32)


def best_build(X):
    Xd, ls = torch.from_numpy(X).cuda(), torch.ones(X.shape[1], device="cuda")
    best = np.inf
    for _ in range(12):
        torch.cuda.synchronize()
        t = time.perf_counter()
        lat = Lattice(Xd, ls)
        best = min(best, time.perf_counter() - t)
        lat.close()
    return best


@pytest.mark.parametrize("lengths", [{0: 64}, {0: 65}, {0: 66}, {0: 62, 7: 70}, {20: 3000},
                                     {0: 1500, 20: 1500}])
def test_products(lengths):
    X = points_with_runs(120, 20, lengths, 3)
    V = synth.gaussian_values(len(X), 5, 9)
    ref = OracleLattice(X, np.ones(20, np.float32))
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, spacing=ref.s)
    assert lat.m == ref.m and lat.sparse_blur
    for blur, mode in (("sequential", 0), ("symmetric", 2)):
        got = lat.mvm(torch.from_numpy(V).cuda(), blur=blur, alpha=0.7).cpu().numpy()
        want = ref.mvm(V.astype(np.float64), mode=mode, alpha=0.7)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), blur


def test_build_time_does_not_follow_the_chain():
    """3000 vertices in one chain against 50 chains of 60: the walks along the former took 1.5
    milliseconds, the rest of the build takes well below one."""
    short = best_build(points_with_runs(400, 20, {0: 60}, 3).repeat(8, axis=0)[:3400])
    long = best_build(points_with_runs(400, 20, {0: 3000}, 3))
    print("build: %.0f us with short chains, %.0f us with a long one" % (short * 1e6, long * 1e6))
    assert long <= 2.0 * short + 300e-6
