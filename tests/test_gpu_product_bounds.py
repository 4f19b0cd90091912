"""The product engines against bounds that a lost operand plane breaks, at every length of the copy ring.

Inputs are complex Gaussian of unit variance per part, so after k terms a real sum has standard deviation
sqrt(2 k), and 5 of them bound its partial sums.
* Split 3xTF32: hi and lo hold 11 bits each, rounded to nearest, so a product of parts is off by at most
  2^-22 (either operand's remainder, and lo lo) each, 3 in all, and the tensor core's sum over a k-step of 8 reals by at
  most 2 more of its terms: 5 2^-22 (|A| |B|)_ij.  The K / 4 sums of k-steps add rounding errors of at most
  2^-24 5 sqrt(2 K), independent and without bias: 6 standard deviations of their sum are 22 K 2^-24.
* FP64 and exact digits: 2 K roundings of at most 2^-53 5 sqrt(2 K) for a real part, as independent:
  6 standard deviations 60 K 2^-53, and as much for numpy's own product.
The CPU test shows that a product from the hi parts of one operand breaks the first bound at every shape.
"""
import ctypes

import numpy as np
import pytest

import workloads

# K: 1 to 4 slabs of 16 (the ring holds 3), ragged ones, and a ring that wraps 80 times
SHAPES = [(300, 130, K) for K in (1, 16, 17, 32, 33, 48, 49, 64, 65, 111, 112, 113)] + [(40, 70, 4000), (2500, 1300, 50)]


def _inputs(M, N, K, opB):
    r = np.random.Generator(np.random.PCG64([workloads.SEED, M, N, K, opB]))
    b = (N, K) if opB else (K, N)
    return (r.standard_normal((M, K)) + 1j * r.standard_normal((M, K)), r.standard_normal(b) + 1j * r.standard_normal(b))


def _reference(A, B, opB):
    return A @ (B.conj().T if opB else B)


def _bound(precision, A, B, opB):
    K = A.shape[1]
    if precision == 1:
        return 5 * 2.0 ** -22 * _reference(np.abs(A), np.abs(B), opB) + 22 * K * 2.0 ** -24
    return 120 * K * 2.0 ** -53


def _hi(x):
    """Parts rounded to 11 significant bits."""
    def cut(v):
        m, e = np.frexp(v)
        return np.ldexp(np.rint(m * 2.0 ** 11), e - 11)
    return cut(x.real) + 1j * cut(x.imag)


@pytest.mark.parametrize("shape", SHAPES)
def test_a_lost_plane_breaks_the_bound(shape):
    A, B = _inputs(*shape, 0)
    ref, bound = _reference(A, B, 0), _bound(1, A, B, 0)
    for bad in (_hi(A) @ B, A @ _hi(B)):
        assert np.any(np.abs((bad - ref).real) > bound)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("opB", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_products_within_their_bounds(lib, precision, opB, shape):
    import torch
    M, N, K = shape
    A, B = _inputs(M, N, K, opB)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    outs = [torch.full((M, N), float("nan"), dtype=torch.complex128, device="cuda") for _ in range(4)]
    for out in outs:  # back to back: the CTAs of one launch follow those of the other on their SMs
        assert lib.tebd_zgemm(precision, opB, M, N, K, 1.0, ctypes.c_void_p(tA.data_ptr()), K,
                              ctypes.c_void_p(tB.data_ptr()), B.shape[1], ctypes.c_void_p(out.data_ptr()), N,
                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    assert all(torch.equal(out, outs[0]) for out in outs[1:])
    err, bound = outs[0].cpu().numpy() - _reference(A, B, opB), _bound(precision, A, B, opB)
    assert np.all(np.abs(err.real) <= bound) and np.all(np.abs(err.imag) <= bound)
