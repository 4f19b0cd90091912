"""The dense gate by total occupation at the local dimensions of its widest variant (6 to 8), against the oracle.

One layer of a saturated state: spectra to 1e-10 and densities to 1e-9, the bounds of single updates.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("d,chi", [(5, 13), (6, 11), (7, 9), (8, 5)])
def test_layer(lib, precision, d, chi):
    from oracle.tebd import TEBD as OracleTEBD
    from paper_2401_05301_gb300 import TEBD
    L, i = 7, 3
    args = (L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 0.5 * (L + 1), 0.02)
    B, lam, _ = workloads.synthetic_state(L, d, chi)
    g = TEBD(*args, precision=precision)
    g.set_state(B, lam)
    g.layer(0, False)
    o = OracleTEBD(*args)
    o.set_state(B, lam)
    o.apply_gate(i, o.gate(i + 1, 0.5 * 0.02))
    dims = g.bond_dims()
    for k in (i + 1, i + 2):
        assert dims[k] == len(o.lam[k])
        assert np.max(np.abs(g.get_lambda(k) - o.lam[k])) < 1e-10
    n, _ = g.measure()
    assert np.max(np.abs(n[i:i + 3] - o.densities()[i:i + 3])) < 1e-9
    g.close()
