"""Three probes run as rows of four columns; the sums of CG keep the shape they have without the
zero column, so the quadratures have the same bits as on a lattice whose padded rows do not fit
(SGP_FAULT=cols_oom:3), as long as the rows are one wave (the slice's grid is what the device
keeps resident, which differs between the two kernels).  One point, one and several blocks of
rows; a launch a pass, one cluster, chains and direction lists; and one to four probes against
the FP64 oracle (1e-3 of the largest, as for the other quadratures)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice, rademacher_sketch
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,order", [(1, 3, 1), (85, 3, 1), (86, 3, 1), (20_000, 6, 1),
                                       (700, 20, 1), (700, 20, 2)])
def test_same_bits_as_without_padding(monkeypatch, n, d, order):
    X = torch.from_numpy(synth.gmm_points(max(n, 2), d, 7)[:n].copy()).cuda()
    Z = torch.from_numpy(rademacher_sketch(n, 3, 3).astype(np.float32)).cuda()
    kw = dict(order=order, kernel="rbf_coverage" if order > 1 else "rbf_binomial")
    got = Lattice(X, 1.0, **kw).logdet(Z, noise=0.5, max_lanczos=20)
    monkeypatch.setenv("SGP_FAULT", "cols_oom:3")
    lat = Lattice(X, 1.0, **kw)
    monkeypatch.delenv("SGP_FAULT")
    want = lat.logdet(Z, noise=0.5, max_lanczos=20)
    assert np.array_equal(got[1], want[1]) and got[0] == want[0]


@pytest.mark.parametrize("probes", [1, 2, 3, 4])
def test_few_probes_match_oracle(probes):
    n, d = 3000, 6
    X = synth.gmm_points(n, d, 6)
    Z = rademacher_sketch(n, probes, 3).astype(np.float32)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0)
    est, quads = lat.logdet(torch.from_numpy(Z).cuda(), noise=0.05, max_lanczos=60)
    est_ref, ref = OracleLattice(X, np.ones(d, np.float32)).logdet(
        Z.astype(np.float64), 0.05, max_lanczos=60)
    assert np.abs(quads - ref).max() <= 1e-3 * np.abs(ref).max()
    assert est == pytest.approx(est_ref, rel=1e-3)
