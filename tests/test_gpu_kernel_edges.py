"""GPU kernels at the sizes where their tiles, pieces and variants change.

* tebd_zgemm on every engine around its tile edges, split reductions and direct tiles, against a
  64-bit product of the same inputs.  Bounds: a complex FP64 or exact-digit product of K terms is off by at
  most 4 K eps max|A| max|B|; 3xTF32 drops 2^-22 of each real product and adds in FP32, below
  K 2^-20 max|A| max|B|.
* one Trotter layer of saturated states whose Gram matrices cross the reduction's piece sizes (256, 512,
  1024 trailing indices), its 64-column tail and the lanes of the bisection, against the dense oracle's
  update of the same triple: spectra to 1e-10 and densities to 1e-9, the bounds of single updates in the
  parity tests.
"""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (16, 16, 16), (17, 33, 16), (24, 24, 96), (128, 64, 16), (129, 65, 17), (40, 7, 4000),
          (250, 100, 32), (1000, 250, 33), (4096, 31, 128)]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("opB", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_zgemm_edges(lib, precision, opB, shape):
    import torch
    M, N, K = shape
    rng = np.random.Generator(np.random.PCG64([workloads.SEED, M, N, K, opB]))
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((N, K) if opB else (K, N)) + 1j * rng.standard_normal((N, K) if opB else (K, N))
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    out = torch.full((M, N), float("nan"), dtype=torch.complex128, device="cuda")
    for alpha in (1.0, -0.75):
        st = lib.tebd_zgemm(precision, opB, M, N, K, alpha, ctypes.c_void_p(tA.data_ptr()), K,
                            ctypes.c_void_p(tB.data_ptr()), B.shape[1], ctypes.c_void_p(out.data_ptr()), N,
                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        ref = alpha * (A @ (B.conj().T if opB else B))
        unit = 2.0 ** -20 if precision == 1 else 4 * 2.0 ** -52
        bound = K * unit * np.abs(A).max() * np.abs(B).max()
        err = np.max(np.abs(out.cpu().numpy() - ref))
        assert err <= bound, (err, bound)


# (d, chi, L): m = chi d of the middle triple, kmax = chi
CUTS = [(2, 16, 12), (2, 33, 14), (3, 43, 12), (3, 86, 12), (4, 129, 12), (2, 257, 20), (4, 257, 12)]


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("d,chi,L", CUTS)
def test_layer_across_piece_sizes(lib, precision, d, chi, L):
    from oracle.tebd import TEBD as OracleTEBD
    from paper_2401_05301_gb300 import TEBD
    args = (L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 0.5 * (L + 1), 0.02)
    B, lam, _ = workloads.synthetic_state(L, d, chi)
    i = 3 * ((L // 2 - 1) // 3)  # a triple of layer A in the middle
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
