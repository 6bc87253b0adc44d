"""The gradients of a product asked for one by one or together: every one has the same bits
whichever others are wanted, dV those of the transposed product, and all agree with the FP64
oracle.  The symmetric backward runs both of its blurs at once as soon as dX or dls is wanted;
lattices with vertices of thousands of points (whose partial sums are combined in a tree), dense,
in one cluster launch, and sparse.

Tolerances as for the other lattice gradients: dV 1e-5, dX and dls 1e-4 relative L2 (fp32); for
bf16 values 1e-2 and, for dX and dls, which are differences of neighbouring vertices' values,
5e-2."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu

SETS = {"crowded": (40_000, 2, 1.0), "crowded3": (30_001, 3, 2.0), "clusters": (3000, 5, 1.0),
        "dense": (20_000, 9, 1.0), "sparse": (400, 20, 1.0)}


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("points", sorted(SETS))
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8, 127])
@pytest.mark.parametrize("values,tols", [("f32", (1e-5, 1e-4, 1e-4)), ("bf16", (1e-2, 5e-2, 5e-2))])
def test_gradients_do_not_depend_on_what_else_is_wanted(points, k, values, tols):
    n, d, scale = SETS[points]
    X = synth.gmm_points(n, d, 11)
    ls = np.full(d, scale, np.float32)
    V, G = synth.gaussian_values(n, k, 12), synth.gaussian_values(n, k, 13)
    lat = Lattice(gpu(X), gpu(ls), value_dtype=values)

    def grads(*want):
        return lat.mvm_backward(gpu(X), gpu(ls), gpu(V), gpu(G), blur="symmetric", alpha=0.9,
                                want=want)

    together = grads("V", "X", "ls")
    assert torch.equal(grads("V")[0], together[0])
    assert torch.equal(lat.mvm(gpu(G), blur="symmetric", alpha=0.9), together[0])
    assert torch.equal(grads("X")[1], together[1])
    assert torch.equal(grads("ls")[2], together[2])
    _, dX, dls = grads("X", "ls")
    assert torch.equal(dX, together[1]) and torch.equal(dls, together[2])
    want = OracleLattice(X, ls).mvm_backward(V.astype(np.float64), G.astype(np.float64), mode=2,
                                             alpha=0.9)
    for name, a, b, tol in zip(("dV", "dX", "dls"), together, want, tols):
        rel = np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
        assert rel <= tol, (name, rel)
