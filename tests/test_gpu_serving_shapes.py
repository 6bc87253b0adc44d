"""Served posteriors at the sizes where the batched iteration changes shape: column counts from
one tile of 8 to four, point counts around the rows of a block (340 of the vectors at 12 columns,
512 of B^T r and 576 of z), more than one round of B^T r partials, and few vertices with very many
points, against the FP64 oracle.

Tolerances as for the other served posteriors: solves to 1e-5, mean to 1e-3 relative L2, variance
to 1e-3 absolute."""

import numpy as np
import pytest

from oracle import gp_posterior
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.serve import Server

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ns,d,probes", [
    (300, 1, 3, 1), (339, 1, 8, 8), (340, 1, 8, 8), (511, 2, 5, 3), (575, 1, 8, 5),
    (576, 1, 8, 11), (577, 16, 20, 14), (1151, 1, 3, 22), (1500, 64, 8, 30), (9000, 64, 2, 8),
    (17000, 8, 3, 8),
])
def test_posterior_at_block_edges(n, ns, d, probes):
    r = synth.serving_stream(1, 100 + n, n_range=(n, n + 1), dims=(d,), test_points=ns)[0]
    tol = 1e-5
    with Server(max_active=2, probes=probes, tol=tol, max_iter=2000, precond_min_kappa=0.0) as srv:
        rid = srv.submit(r["X"], r["y"], r["Xs"], r["lengthscales"], r["outputscale"], r["noise"],
                         r["seed"])
        srv.run_until_idle()
        mean, var = srv.result(rid)
        st = srv.stats(rid)
    m_ref, v_ref, _, _ = gp_posterior(r["X"], r["y"], r["Xs"], r["lengthscales"], r["noise"],
                                      probes=probes, seed=r["seed"], tol=tol, max_iter=2000,
                                      precond_rank=st["precond_rank"])
    assert st["status"] == 0 and st["rel_res"] <= tol and st["precond_rank"] > 0
    assert np.linalg.norm(mean - m_ref) <= 1e-3 * np.linalg.norm(m_ref)
    assert np.abs(var - v_ref).max() <= 1e-3
