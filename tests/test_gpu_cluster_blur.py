"""Small lattices blurred in one launch by thread-block clusters: vertex counts around one
vertex, the rows of a block and the largest lattice taken, column counts around the number of
clusters, both stencil orders taken and one beyond, against the FP64 oracle; and the products
of a CG.  Tolerance as for the other products: 1e-5 relative L2 (fp32), 1e-2 (bf16)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def compare(X, k, order=1, values="f32", tol=1e-5):
    n, d = X.shape
    V = synth.gaussian_values(n, k, 4)
    ref = OracleLattice(X, np.ones(d, np.float32), 1 if order > 1 else 0, order)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, spacing=ref.s, order=order, value_dtype=values,
                  kernel="rbf_coverage" if order > 1 else "rbf_binomial")
    assert lat.m == ref.m
    for blur, mode in (("sequential", 0), ("transpose", 1), ("symmetric", 2)):
        got = lat.mvm(torch.from_numpy(V).cuda(), blur=blur, beta=0.3).cpu().numpy()
        want = ref.mvm(V.astype(np.float64), mode=mode, beta=0.3)
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), (lat.m, blur)
    return lat.m


@pytest.mark.parametrize("spread,n", [(0.0, 5), (0.05, 50), (0.6, 400), (1.0, 700), (1.0, 2600),
                                      (1.0, 6000), (1.0, 9000)])
@pytest.mark.parametrize("k", [1, 2, 4, 13])
def test_vertex_counts(spread, n, k):
    """From one simplex (5 vertices) through the rows of one block (64) to beyond the 16,384
    vertices of the largest cluster."""
    m = compare(np.float32(spread) * synth.gmm_points(n, 4, 8) * np.float32(3.0), k)
    assert m >= 5


@pytest.mark.parametrize("k", [28, 32, 33, 36])
def test_column_groups(k):
    compare(synth.gmm_points(800, 3, 8), k)


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("values,tol", [("f32", 1e-5), ("bf16", 1e-2)])
def test_stencil_orders(order, values, tol):
    compare(synth.gmm_points(3000, 3, 8), 5, order, values, tol)


@pytest.mark.parametrize("values", ["f32", "bf16"])
def test_same_bits_as_one_launch_a_pass(values):
    """33 columns take a launch a pass, 32 of them the clusters: the shared columns agree."""
    X = synth.gmm_points(1500, 5, 2)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, value_dtype=values)
    V = torch.from_numpy(synth.gaussian_values(1500, 36, 3)).cuda()
    for blur in ("sequential", "symmetric"):
        wide = lat.mvm(V, blur=blur)
        narrow = lat.mvm(V[:, :32].contiguous(), blur=blur)
        assert torch.equal(wide[:, :32], narrow)
