"""Log-determinant quadrature at the edges of its ranges: one step, two, a count that is not
a multiple of a warp, the largest; one probe, a few, the largest probe count."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice, rademacher_sketch
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps,probes", [(1, 1), (2, 5), (33, 3), (256, 2), (7, 256)])
def test_quadrature_edges(steps, probes):
    """tol 0 runs every step.  The products' fp32 rounding (1e-6 relative) enters the
    quadrature once per step while the recurrence stays orthogonal (up to 33 steps at noise
    0.5); beyond, the bound of the 100-step comparison (1e-3) applies."""
    n, d, noise = 900, 4, 0.5
    X = synth.gmm_points(n, d, 11)
    Z = rademacher_sketch(n, probes, 5).astype(np.float32)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0)
    est, quads = lat.logdet(torch.from_numpy(Z).cuda(), noise=noise, max_lanczos=steps, tol=0.0)
    est_ref, ref = OracleLattice(X, np.ones(d, np.float32)).logdet(
        Z.astype(np.float64), noise, max_lanczos=steps, tol=0.0)
    scale = np.abs(ref).max()
    assert np.abs(quads - ref).max() <= (1e-4 if steps <= 33 else 1e-3) * scale
    assert abs(est - est_ref) <= (1e-4 if steps <= 33 else 1e-3) * scale
