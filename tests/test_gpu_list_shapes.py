"""Blurs through the direction lists with few columns: a thread a column or a thread a row, by the
column count and the length of the list (both sides of its line, 65,536 vertices).  The columns
have the same bits as in a product of eight columns, which agrees with the FP64 oracle where the
lists are short (1e-5 relative L2 for fp32 values, ~1e-6 expected; 1e-2 for bf16)."""

import ctypes

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import _lib, synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def mean_list(lat):
    sparse, pairs = ctypes.c_int(), ctypes.c_int64()
    assert _lib.load().sgp_lattice_blur_lists(lat._h, ctypes.byref(sparse), ctypes.byref(pairs)) == 0
    return pairs.value / (lat.d + 1)


@pytest.mark.parametrize("n,d,order,long", [(300, 20, 2, False), (2000, 33, 3, False),
                                            (45_000, 20, 2, True)])
@pytest.mark.parametrize("values,tol", [("f32", 1e-5), ("bf16", 1e-2)])
def test_columns(n, d, order, long, values, tol):
    X = synth.gmm_points(n, d, 7)
    V = synth.gaussian_values(n, 8, 9)
    ref = None if long else OracleLattice(X, np.ones(d, np.float32), 1, order)
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0, kernel="rbf_coverage", order=order,
                  spacing=0.0 if long else ref.s, value_dtype=values)
    assert lat.sparse_blur and (mean_list(lat) > 1 << 16) == long
    Vd = torch.from_numpy(V).cuda()
    for blur, mode in (("symmetric", 2), ("sequential", 0)):
        full = lat.mvm(Vd, blur=blur)
        if ref is not None:
            want = ref.mvm(V.astype(np.float64), mode=mode)
            assert np.linalg.norm(full.cpu().numpy() - want) <= tol * np.linalg.norm(want), blur
        for k in (1, 2, 3, 4, 5):
            assert torch.equal(lat.mvm(Vd[:, :k].contiguous(), blur=blur), full[:, :k]), (blur, k)
