"""Log determinants whose probes or operators leave the quadrature without a value."""

import ctypes

import numpy as np
import pytest
import torch

from oracle import rademacher_sketch
from paper_2106_06695_gb300 import _lib, synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def logdet(lat, Z, noise, steps, tol=0.0):
    """(status, estimate, per-probe values) of the C entry point."""
    est, quads = ctypes.c_double(), np.full(Z.shape[1], -1.0)
    status = _lib.load().sgp_logdet(lat._handle(), Z.data_ptr(), Z.shape[1], noise, steps, tol,
                                    ctypes.byref(est), quads.ctypes.data)
    return status, est.value, quads


@pytest.mark.parametrize("probes,bad", [(3, 1), (8, 7), (1, 0)])
@pytest.mark.parametrize("value", [np.nan, np.inf, 3e38])
def test_a_probe_without_iterations_counts_as_zero(probes, bad, value):
    """A column that CG cannot step on (not finite, or its squares overflow) has no tridiagonal:
    its value is 0, the others keep their bits."""
    X = torch.from_numpy(synth.gmm_points(500, 3, 5)).cuda()
    lat = Lattice(X, 1.0)
    Z = torch.from_numpy(rademacher_sketch(500, probes, 3).astype(np.float32)).cuda()
    status, _, good = logdet(lat, Z, 0.1, 30)
    assert status == 0
    Z[7, bad] = value
    status, est, quads = logdet(lat, Z, 0.1, 30)
    assert status == 0 and quads[bad] == 0.0
    assert np.array_equal(np.delete(quads, bad), np.delete(good, bad))
    assert est == pytest.approx(quads.mean(), rel=1e-14)
