"""Small lattices on a device that cannot hold a 16-block cluster (SGP_FAULT=no_cluster answers the
occupancy query so): products, gradients, solves and log determinants, the last two inside a
captured graph, take a launch a pass and give the same bits."""

import numpy as np
import pytest
import torch

from paper_2106_06695_gb300 import _lib, synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("values", ["f32", "bf16"])
@pytest.mark.parametrize("order,k", [(1, 1), (1, 2), (1, 9), (2, 5)])
def test_same_results_without_clusters(monkeypatch, order, k, values):
    n, d = 1500, 5
    X = gpu(synth.gmm_points(n, d, 2))
    V, G = gpu(synth.gaussian_values(n, k, 3)), gpu(synth.gaussian_values(n, k, 4))
    Z = torch.sign(V)
    kw = dict(order=order, kernel="rbf_coverage" if order > 1 else "rbf_binomial",
              value_dtype=values)
    lib = _lib.load()

    def results(lat):
        before = lib.sgp_kernel_launches()
        out = [lat.mvm(V, blur=b) for b in ("symmetric", "sequential")]
        launches = lib.sgp_kernel_launches() - before
        out += list(lat.mvm_backward(X, 1.0, V, G, blur="symmetric"))
        x, iters, rel = lat.cg(V, noise=0.1, tol=1e-3, max_iter=30)
        out += [x, torch.from_numpy(iters), torch.from_numpy(rel)]
        est, quad = lat.logdet(Z, noise=0.1, max_lanczos=20)
        return out + [torch.tensor(est), torch.from_numpy(quad)], launches

    with_clusters, few = results(Lattice(X, 1.0, **kw))
    monkeypatch.setenv("SGP_FAULT", "no_cluster")
    lat = Lattice(X, 1.0, **kw)
    monkeypatch.delenv("SGP_FAULT")
    without, many = results(lat)
    assert many - few == 3 * (d + 1) - 2  # 2 (d + 1) and d + 1 passes instead of one launch each
    for a, b in zip(with_clusters, without):
        assert torch.equal(a, b)
