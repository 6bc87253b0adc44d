"""Products whose column count is not a multiple of 4 (rows padded with zero columns inside
the operator), caller buffers off 16-byte alignment, and the shift beta V, against the FP64
oracle: dense, sparse and many-points-per-vertex lattices, fp32 and bf16 values.

Tolerances: 1e-5 relative L2 for fp32 values (about 2^-24 per operation, random-signed, over
the splat, 2 (d + 1) passes and the slice: 1e-6 expected), 1e-2 for bf16 ones (2^-9 per stored
value over up to 2 (d + 1) + 1 stores: 6e-3 at d = 3, 8; lazily scaled rows store fewer)."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu

SETS = {"dense": (1501, 8), "sparse": (300, 50), "crowded": (40_003, 3)}


def offset(a):
    """A CUDA copy of the array whose rows start 4 bytes off 16-byte alignment."""
    buf = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    t = buf[1:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("points", sorted(SETS))
@pytest.mark.parametrize("k", [1, 2, 3, 5, 9, 14, 16])
def test_product_with_any_column_count(points, k):
    n, d = SETS[points]
    X = synth.gmm_points(n, d, 21)
    V = synth.gaussian_values(n, k, 21)
    ref = OracleLattice(X, np.ones(d, np.float32))
    for values, tol in (("f32", 1e-5), ("bf16", 1e-2)):
        lat = Lattice(torch.from_numpy(X).cuda(), 1.0, value_dtype=values)
        for blur, mode, beta in (("symmetric", 2, 0.25), ("transpose", 1, 0.0)):
            want = ref.mvm(V.astype(np.float64), mode=mode, alpha=0.5, beta=beta)
            for shift in (False, True):
                Vd = offset(V) if shift else torch.from_numpy(V).cuda()
                out = offset(np.zeros_like(V)) if shift else None
                got = lat.mvm(Vd, blur=blur, alpha=0.5, beta=beta, out=out).cpu().numpy()
                rel = np.linalg.norm(got - want) / np.linalg.norm(want)
                assert rel <= tol, (values, blur, shift, rel)


def test_columns_do_not_depend_on_their_neighbours():
    """Column c of a 16-column product equals the same column of a 3- and a 12-column one (no
    vertex here is long enough for the column count to shape its sum)."""
    X = synth.gmm_points(1501, 8, 22)
    V = torch.from_numpy(synth.gaussian_values(1501, 16, 22)).cuda()
    lat = Lattice(torch.from_numpy(X).cuda(), 1.0)
    full = lat.mvm(V, blur="symmetric")
    for k in (3, 12):
        assert torch.equal(lat.mvm(V[:, :k].contiguous(), blur="symmetric"), full[:, :k])
