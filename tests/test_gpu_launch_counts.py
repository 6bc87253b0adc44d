"""sgp_kernel_launches against a count by hand of a served request's kernels."""

import numpy as np
import pytest
import torch

from paper_2106_06695_gb300 import _lib, synth
from paper_2106_06695_gb300.lattice import Lattice
from paper_2106_06695_gb300.serve import Server

pytestmark = pytest.mark.gpu


def served(request, **kw):
    """(kernels outside the iterations, kernels of an iteration) of a request that stops at
    once: one round of `check_every` iterations, run with 1 and with 2."""
    counts = []
    for rounds in (1, 2):
        with Server(max_active=1, max_iter=0, check_every=rounds, precond_min_kappa=0.0,
                    **kw) as srv:
            before = _lib.load().sgp_kernel_launches()
            i = srv.submit(request["X"], request["y"], request["Xs"], request["lengthscales"],
                           seed=request["seed"])
            srv.run_until_idle()
            counts.append(_lib.load().sgp_kernel_launches() - before)
            assert srv.stats(i)["status"] == 0
    return 2 * counts[0] - counts[1], counts[1] - counts[0]


@pytest.mark.parametrize("rank,probes", [(100, 8), (16, 2)])
def test_preconditioned_request(rank, probes):
    r = synth.serving_stream(1, 5, n_range=(3000, 3001), dims=(3,), test_points=32)[0]
    plain, step = served(r, precond_rank=0, probes=probes)
    pre, pre_step = served(r, precond_rank=rank, probes=probes)
    # splat, its fix-up, 2 (d + 1) passes, slice, alpha, x and r, check and beta, p
    assert step == 7 + 2 * 4
    # B^T r, its sums, Minv times them, z
    assert pre_step == step + 4
    kp = (probes + 2 + 3) // 4 * 4
    P = np.concatenate([r["X"], r["Xs"]])
    lat = Lattice(torch.from_numpy(np.ascontiguousarray(P, np.float32)).cuda(),
                  torch.from_numpy(np.asarray(r["lengthscales"], np.float32)))
    V = torch.ones(len(P), kp, device="cuda")
    before = _lib.load().sgp_kernel_launches()
    lat.mvm(V, blur="symmetric")
    product = _lib.load().sgp_kernel_launches() - before - 1  # without the caller's permutation
    # condition estimate, per group of kp sketch columns fill, product and gather, two Gram
    # matrices (2 each), two Cholesky factors, the rows' product, two inverses; then z of r
    chunks = -(-rank // kp)
    assert pre - plain == 1 + chunks * (2 + product) + 9 + 4
