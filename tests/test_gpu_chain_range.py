"""Sparse fp32 products over the whole exponent range: their chains hold values divided by powers
of the centre tap, which must neither overflow nor underflow where the product itself does not.
Magnitudes near both ends of fp32, in V and in alpha, at the default spacing and at a small one
(centre tap 0.6 instead of 0.94, so a factor of 3e22 over the passes of d = 50), up to the most
passes there are.

Tolerance as for the other products: 1e-5 relative L2; a power of two changes no bit of it as
long as no value is denormal, and those are 2^-24 of the typical one or less here."""

import numpy as np
import pytest
import torch

from oracle import OracleLattice
from paper_2106_06695_gb300 import synth
from paper_2106_06695_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("d,k", [(20, 5), (50, 9), (63, 1), (90, 4), (127, 2)])
@pytest.mark.parametrize("spacing", [0.0, 0.25])
@pytest.mark.parametrize("blur,mode", [("symmetric", 2), ("sequential", 0)])
def test_magnitudes(d, k, spacing, blur, mode):
    n = 60
    X = synth.gmm_points(n, d, 5)
    ls = np.ones(d, np.float32)
    V, G = synth.gaussian_values(n, k, 9), synth.gaussian_values(n, k, 10)
    if spacing == 0.0:
        spacing = OracleLattice(X, ls).s
    ref = OracleLattice(X, ls, spacing=spacing)
    lat = Lattice(gpu(X), gpu(ls), spacing=ref.s)
    assert lat.m == ref.m and lat.sparse_blur
    want = ref.mvm(V.astype(np.float64), mode=mode)
    norm = np.linalg.norm(want)

    def close(got, power):
        a = np.ldexp(got.cpu().numpy().astype(np.float64), -power)
        assert np.linalg.norm(a - want) <= 1e-5 * norm, power

    # results of 2^-100 or more at the low end (0.6^256 of what a vertex receives stays there at
    # the most passes: V itself has to be large then)
    low = int(max(-90, np.ceil(-100 - np.log2(norm / np.sqrt(want.size)))))
    base = max(0, low)
    close(lat.mvm(gpu(np.ldexp(V, base)), blur=blur), base)
    for power in (110, low):
        big = gpu(np.ldexp(V, power))
        close(lat.mvm(big, blur=blur), power)
        close(lat.mvm(gpu(np.ldexp(V, base)), blur=blur, alpha=2.0 ** (power - base)), power)
        close(lat.mvm(big, blur=blur, alpha=2.0 ** (base - power)), base)
    # dV = alpha W B^T W^T G, alone and with the other gradients
    want = ref.mvm(G.astype(np.float64), mode=(1 if mode == 0 else 2))
    norm = np.linalg.norm(want)
    for wanted in (("V",), ("V", "X")):
        got, _, _ = lat.mvm_backward(gpu(X), gpu(ls), gpu(V), gpu(np.ldexp(G, 110)), blur=blur,
                                     alpha=2.0 ** (base - 110), want=wanted)
        close(got, base)
