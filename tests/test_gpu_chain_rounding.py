"""BF16 rows of sparse lattices, blurred by chains, round where the direction lists round them:
a stored row is the value over the centre taps since the pass that last wrote it.  Against an
emulation of that scheme on the host.

Tolerance: the emulation sums in another order, so an fp32 difference of about 1e-7 of a row's
neighbours flips the rounding of a value (2^-8) with a probability of about 3e-5 a pass: after 2 D =
42 to 102 passes a relative L2 of 4e-3 sqrt(102 * 3e-5) = 2.2e-4 at most, doubled.  Rows rounded at
other places are 1.6e-3 away."""

import numpy as np
import pytest
import torch

from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def bf16(a):
    return torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16).to(torch.float32).numpy()


def emulate(lat, V, half):
    e = lat.export()
    keys, idx, w = e["keys"].astype(np.int64), e["idx"], e["w"].astype(np.float64)
    m, D = keys.shape
    where = {tuple(r): i for i, r in enumerate(keys)}
    g0, g1 = float(np.float32(half[0])), float(np.float32(half[1]))
    pw = np.float32(half[0] ** np.arange(2 * D + 1)).astype(np.float64)
    x = np.zeros((m, V.shape[1]))
    for c in range(D):
        np.add.at(x, idx[:, c], w[:, c:c + 1] * V.astype(np.float64))
    x = np.vstack([bf16(x), np.zeros((1, V.shape[1]))]).astype(np.float64)  # last row: absent
    epoch = np.zeros(m + 1, np.int64)
    links = []
    for j in range(D):
        u = -np.ones(D, np.int64)
        u[j] += D
        links.append([np.array([where.get(tuple(r), m) for r in keys + s * u]) for s in (-1, 1)])
    for t in range(2 * D):
        a, b = links[t if t < D else 2 * D - 1 - t]
        act = np.flatnonzero((a < m) | (b < m))
        value = lambda v: np.float32(pw[t - epoch[v]][:, None] * x[v]).astype(np.float64)
        new = g0 * value(act) + g1 * np.float32(value(a[act]) + value(b[act]))
        x[act], epoch[act] = bf16(new), t + 1
    x = bf16(pw[2 * D - epoch][:, None] * x).astype(np.float64)
    return (w[:, :, None] * x[idx]).sum(1)


@pytest.mark.parametrize("n,d,k", [(300, 20, 3), (200, 33, 8), (150, 50, 9)])
def test_bf16_chains_round_as_direction_lists(n, d, k):
    X = synth.gmm_points(n, d, 41)
    V = synth.gaussian_values(n, k, 42)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, value_dtype="bf16")
    assert lat.sparse_blur
    got = lat.mvm(torch.from_numpy(V).cuda(), blur="symmetric").cpu().numpy()
    want = emulate(lat, V, lat.stencil()[2])
    print("relative L2 %.1e" % (np.linalg.norm(got - want) / np.linalg.norm(want)))
    assert np.linalg.norm(got - want) <= 4.4e-4 * np.linalg.norm(want)
