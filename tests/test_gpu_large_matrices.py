"""Matrices large enough for the eigen-solver's last variants, at the largest local dimension.

Triple 4 of an L = 8, d = 8 chain has m = 8 chi rows and few columns (at most 512), so the oracle's SVD stays cheap:
chi = 261 (m = 2088) crosses the reduction's last piece sizes at 2048 trailing indices, and with 769 eight warps share an
eigenvector of the first cut's FP64 back-transformation (m = 6152) and four of the second's (4096).
Bounds: those of single updates, spectra to 1e-10 and densities to 1e-9.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [261, 769])
def test_layer_of_a_tall_triple(lib, chi):
    from oracle.tebd import TEBD as OracleTEBD
    from paper_2401_05301_gb300 import TEBD
    L, d, i = 8, 8, 4
    args = (L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 0.5 * (L + 1), 0.02)
    B, lam, _ = workloads.synthetic_state(L, d, chi)
    o = OracleTEBD(*args)
    o.set_state(B, lam)
    o.apply_gate(i, o.gate(i + 1, 0.5 * 0.02))
    for precision in (0, 2):
        g = TEBD(*args, precision=precision)
        g.set_state(B, lam)
        g.layer(1, False)
        dims = g.bond_dims()
        for k in (i + 1, i + 2):
            assert dims[k] == len(o.lam[k]), precision
            assert np.max(np.abs(g.get_lambda(k) - o.lam[k])) < 1e-10, precision
        n, _ = g.measure()
        assert np.max(np.abs(n[i:i + 3] - o.densities()[i:i + 3])) < 1e-9, precision
        g.close()
