"""Calls on a lattice when device memory is short.  SGP_FAULT=cols_oom:<c> makes the library's
allocations of more than c columns fail on the host, before any device work.

Tolerance as for the other products: 1e-5 relative L2 (fp32 values, ~1e-6 expected)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
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
