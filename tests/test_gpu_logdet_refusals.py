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


@pytest.mark.parametrize("probes", [6, 64])
@pytest.mark.parametrize("n,d,ls,steps", [(5000, 3, 5.0, 200), (500, 2, 2.0, 256),
                                          (50, 2, 10.0, 256), (50, 2, 10.0, 100)])
def test_singular_operators_are_refused(n, d, ls, steps, probes):
    """Without noise, more points than vertices: CG runs on past the operator's range and the
    smallest eigenvalues of its tridiagonals are rounding errors of either sign.  Of the probes'
    tridiagonals some come out at zero or below; their values are NaN and the call is refused."""
    X = torch.from_numpy(synth.gmm_points(n, d, 5)).cuda()
    lat = Lattice(X, ls)
    assert lat.m < n
    Z = torch.from_numpy(np.sign(synth.gaussian_values(n, probes, 3))).cuda()
    status, est, quads = logdet(lat, Z, 0.0, steps)
    assert status == 5 and np.isnan(quads).any() and np.isnan(est)


@pytest.mark.parametrize("noise", [1e-6, 1e-3, 1.0])
def test_regular_operators_are_not(noise):
    """The smallest eigenvalue is the noise: above 1e-12 of the largest (1e2 to 1e4 here)."""
    X = torch.from_numpy(synth.gmm_points(5000, 3, 5)).cuda()
    lat = Lattice(X, 5.0)
    Z = torch.from_numpy(rademacher_sketch(5000, 64, 3).astype(np.float32)).cuda()
    status, est, quads = logdet(lat, Z, noise, 200)
    assert status == 0 and np.isfinite(quads).all() and np.isfinite(est)
