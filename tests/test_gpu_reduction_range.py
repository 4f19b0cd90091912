"""The eigen-solver over the range of a double: Gram matrices that are graded over hundreds of decades,
nearly empty, or of a state that is not normalised, against the oracle's update of the same triple.

Each case takes one Trotter layer of a synthetic saturated state whose bond vector left of the middle triple is
multiplied by `scale`, and the second half of it (in the blocked form, the charges up to 3) by
`tail` on top, so its Gram matrix has a trace of about scale^2 and a block of about (scale tail)^2.  The oracle
takes LAPACK's SVD of theta'.  The kept spectra are renormalised by the truncation, so the bounds of single
updates of normalised states apply to them as they stand: 1e-10.  The densities of the triple's last two sites
(left of which the bond vectors are the renormalised ones) hold to 1e-9.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

# (d, chi, L): m = chi d rows, below and above the 64 that one block reduces alone
SIZES = [(4, 12, 8), (2, 40, 14), (3, 43, 14), (4, 86, 14)]
RANGES = [(1.0, 1e-90), (1.0, 1e-48), (1e-80, 1.0), (1e-29, 1e-60), (1e29, 1e-150), (1e-2, 1.0), (1e60, 1.0)]


def _middle(L):
    return 3 * ((L // 2 - 1) // 3)  # the triple of layer A in the middle


def _check(g, o, i):
    dims = g.bond_dims()
    for k in (i + 1, i + 2):
        assert dims[k] == len(o.lam[k])
        assert np.max(np.abs(np.sort(g.get_lambda(k)) - np.sort(o.lam[k]))) < 1e-10
    n, _ = g.measure()
    assert np.max(np.abs(n[i + 1:i + 3] - o.densities()[i + 1:i + 3])) < 1e-9


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("scale,tail", RANGES)
@pytest.mark.parametrize("d,chi,L", SIZES)
def test_dense_layer(lib, precision, scale, tail, d, chi, L):
    from oracle.tebd import TEBD as OracleTEBD
    from paper_2401_05301_gb300 import TEBD
    args = (L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 0.5 * (L + 1), 0.02)
    B, lam, _ = workloads.synthetic_state(L, d, chi)
    i = _middle(L)
    lam[i] = lam[i] * scale
    lam[i][len(lam[i]) // 2:] *= tail
    g = TEBD(*args, precision=precision)
    g.set_state(B, lam)
    g.layer(0, False)
    o = OracleTEBD(*args)
    o.set_state(B, lam)
    o.apply_gate(i, o.gate(i + 1, 0.5 * 0.02))
    _check(g, o, i)
    g.close()


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("scale,tail", RANGES)
def test_blocked_layer(lib, precision, scale, tail):
    from oracle.u1 import U1TEBD
    from paper_2401_05301_gb300 import TEBD
    L, d, chi = 14, 4, 600
    args = (L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 0.5 * (L + 1), 0.02)
    B, lam, q = workloads.synthetic_state_u1(L, d, chi, L // 2)
    i = _middle(L)
    lam[i] = np.where(q[i] <= 3, lam[i] * scale * tail, lam[i] * scale)
    g = TEBD(*args, precision=precision, u1=True)
    g.set_state(B, lam)
    g.set_charges(q)
    g.layer(0, False)
    o = U1TEBD(*args)
    o.set_state(B, lam, q)
    o.apply_gate(i, o.gate(i + 1, 0.5 * 0.02))
    _check(g, o, i)
    g.close()
