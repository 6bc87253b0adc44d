"""Calls on a lattice when device memory is short.  SGP_FAULT=cols_oom:<c> makes the library's
allocations of more than c columns fail on the host, before any device work.

Tolerance as for the other products: 1e-5 relative L2 (fp32 values, ~1e-6 expected)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice, rademacher_sketch
from paper_2106_06695_gb300 import SGPError, synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def limited(monkeypatch, columns, X, **kw):
    monkeypatch.setenv("SGP_FAULT", "cols_oom:%d" % columns)
    lat = Lattice(gpu(X), 1.0, **kw)
    monkeypatch.delenv("SGP_FAULT")
    return lat


def check(lat, ref, k):
    V = synth.gaussian_values(lat.n, k, 9)
    got = lat.mvm(gpu(V), blur="symmetric", alpha=0.7).cpu().numpy()
    want = ref.mvm(V.astype(np.float64), mode=2, alpha=0.7)
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), k


@pytest.mark.parametrize("n,d,order", [(1500, 8, 1), (200, 30, 2), (300, 20, 1)])
@pytest.mark.parametrize("k", [3, 9])
def test_product_without_room_for_padding(monkeypatch, n, d, order, k):
    """Dense, direction lists, chains: k columns fit, k rounded up to a multiple of 4 do not."""
    X = synth.gmm_points(n, d, 7)
    ref = OracleLattice(X, np.ones(d, np.float32), 1 if order > 1 else 0, order)
    kw = dict(kernel="rbf_coverage" if order > 1 else "rbf_binomial", order=order, spacing=ref.s)
    lat = limited(monkeypatch, k, X, **kw)
    check(lat, ref, k)
    check(lat, ref, 1)
    with pytest.raises(SGPError) as e:
        check(lat, ref, k + 1)
    assert e.value.status == 2
    check(lat, ref, k)


def test_narrow_product_after_a_failed_wide_one(monkeypatch):
    """The buffer of one pass over the direction lists is given back before a larger one is
    asked for: after that has failed, a narrower product has to ask again."""
    X = synth.gmm_points(200, 30, 7)
    ref = OracleLattice(X, np.ones(30, np.float32), 1, 2)
    lat = limited(monkeypatch, 4, X, kernel="rbf_coverage", order=2, spacing=ref.s)
    assert lat.sparse_blur
    check(lat, ref, 2)
    with pytest.raises(SGPError) as e:
        check(lat, ref, 9)
    assert e.value.status == 2
    for k in (1, 2, 4):
        check(lat, ref, k)


@pytest.mark.parametrize("n,d,k,columns", [
    (1500, 8, 3, 3), (1500, 8, 9, 9),  # dense: neither pairs nor padded rows fit
    (1500, 8, 9, 12),                  # padded rows fit, pairs do not
    (1500, 8, 8, 8), (300, 20, 8, 8), (300, 20, 5, 5),
])
@pytest.mark.parametrize("blur,mode", [("symmetric", 2), ("sequential", 0)])
def test_gradients_without_room_for_padding(monkeypatch, n, d, k, columns, blur, mode):
    """Tolerances as for the other lattice gradients: dV 1e-5, dX and dls 1e-4."""
    X = synth.gmm_points(n, d, 7)
    V, G = synth.gaussian_values(n, k, 9), synth.gaussian_values(n, k, 10)
    ls = np.ones(d, np.float32)
    ref = OracleLattice(X, ls)
    lat = limited(monkeypatch, columns, X, spacing=ref.s)
    got = lat.mvm_backward(gpu(X), gpu(ls), gpu(V), gpu(G), blur=blur, alpha=0.9)
    want = ref.mvm_backward(V.astype(np.float64), G.astype(np.float64), mode=mode, alpha=0.9)
    for a, b, tol in zip(got, want, (1e-5, 1e-4, 1e-4)):
        assert np.linalg.norm(a.cpu().numpy() - b) <= tol * np.linalg.norm(b)
    with pytest.raises(SGPError) as e:
        lat.mvm_backward(gpu(X), gpu(ls), gpu(np.ones((n, 13))), gpu(np.ones((n, 13))), blur=blur)
    assert e.value.status == 2
    check(lat, ref, k)


@pytest.mark.parametrize("n,d", [(1500, 8), (300, 20)])
@pytest.mark.parametrize("k", [3, 5])
def test_log_determinant_without_room_for_padding(monkeypatch, n, d, k):
    """Bounds as for the other quadratures: 1e-3 of the largest, the estimate 1e-4."""
    X = synth.gmm_points(n, d, 6)
    Z = rademacher_sketch(n, k, 3).astype(np.float32)
    ref = OracleLattice(X, np.ones(d, np.float32))
    lat = limited(monkeypatch, k, X, spacing=ref.s)
    est, quads = lat.logdet(gpu(Z), noise=0.05, max_lanczos=60, tol=1e-6)
    est_ref, q_ref = ref.logdet(Z.astype(np.float64), 0.05, max_lanczos=60, tol=1e-6)
    assert np.abs(quads - q_ref).max() <= 1e-3 * np.abs(q_ref).max()
    assert est == pytest.approx(est_ref, rel=1e-4)
    with pytest.raises(SGPError) as e:
        lat.logdet(gpu(np.ones((n, k + 1))), noise=0.05)
    assert e.value.status == 2
