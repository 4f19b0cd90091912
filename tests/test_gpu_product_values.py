"""The product engines on values at the ends of a double's range.

The exact-digit engine is held bitwise against its own definition in integers: a row's parts are rounded to
multiples of 2^(e - 56) (half to even; e: the power of two above the row's largest part), cut into eight balanced
base-128 digits, the pairs of digits s + t <= 7 are summed exactly, and the sum is rounded once to FP64.  Rows with
halves to round, subnormal parts, parts that vanish beside the row's largest, zeros and parts of 1e308 are among them.
A NaN or an infinity spoils its own row (or column) and no other, on every engine; so does, in split 3xTF32,
a part beyond FP32's range.
"""
import ctypes
import math
from fractions import Fraction

import numpy as np
import pytest

import workloads


def _exponent(row):
    m = max(max(abs(z.real), abs(z.imag)) for z in row)
    return max(math.frexp(m)[1], -1021) if m > 0.0 else -1021


def _digits(x, e):
    scaled = abs(Fraction(x)) * Fraction(2) ** (56 - e)
    f = round(scaled)  # half to even
    out = []
    for _ in range(7):
        r = (f + 64) % 128 - 64
        out.append(r)
        f = (f - r) // 128
    out.append(f)
    return [(-d if math.copysign(1.0, x) < 0 else d) for d in reversed(out)]  # most significant first


def _digit_product(A, B):
    """A (M x K) times B (K x N) by the definition above."""
    M, K = A.shape
    N = B.shape[1]
    ea, eb = [_exponent(A[i]) for i in range(M)], [_exponent(B[:, j]) for j in range(N)]
    da = np.array([[[_digits(A[i, k].real, ea[i]), _digits(A[i, k].imag, ea[i])] for k in range(K)] for i in range(M)])
    db = np.array([[[_digits(B[k, j].real, eb[j]), _digits(B[k, j].imag, eb[j])] for k in range(K)] for j in range(N)])
    out = np.empty((M, N), dtype=complex)

    def value(i, j, terms):
        total = 0
        for s in range(8):
            for t in range(8 - s):
                total += sum(sign * int(da[i, :, p, s] @ db[j, :, q, t]) for p, q, sign in terms) << (49 - 7 * (s + t))
        try:
            return float(Fraction(total) * Fraction(2) ** (ea[i] + eb[j] - 63))
        except OverflowError:
            return math.copysign(math.inf, total)

    for i in range(M):
        for j in range(N):
            out[i, j] = complex(value(i, j, ((0, 0, 1), (1, 1, -1))), value(i, j, ((0, 1, 1), (1, 0, 1))))
    return out


def _rows(K, seed):
    """Rows of K complex values, one kind each."""
    r = np.random.Generator(np.random.PCG64([workloads.SEED, 77, K, seed]))

    def z(n=K):
        return r.standard_normal(n) + 1j * r.standard_normal(n)

    half = (2.0 * r.integers(-2 ** 20, 2 ** 20, K) + 1.0) * 2.0 ** -57  # odd multiples of half a unit beside 0.75
    rows = [z(), z() * 1e-300, z() * 1e300 / 4, z() * 4.9e-324 * r.integers(1, 1 << 30, K),
            z() * 10.0 ** r.uniform(-30, 0, K), np.zeros(K, complex), half + 1j * half[::-1], z() * 2.0 ** -1023]
    rows[1][K // 2] = 1e-322
    rows[2][0] = 1e308
    rows[4][K - 1] = -1.0 + 0.5j
    rows[6][0] = 0.75
    rows.append(np.where(np.arange(K) % 3 == 0, -0.0, 1.0 - 2.0 ** -53) + 0j)
    return np.array(rows)


def test_the_definition_is_a_product():
    A, B = _rows(6, 0), _rows(6, 1).T
    for i in (0, 4, 6, 8):
        for j in (0, 4, 6, 8):
            re = sum(Fraction(a.real) * Fraction(b.real) - Fraction(a.imag) * Fraction(b.imag) for a, b in zip(A[i], B[:, j]))
            bound = 6 * 2.0 ** -50 * np.max(np.abs(A[i])) * np.max(np.abs(B[:, j]))
            assert abs(_digit_product(A[i:i + 1], B[:, j:j + 1])[0, 0].real - float(re)) <= bound


def _gpu(lib, precision, opB, A, B, alpha=1.0):
    import torch
    Bm = np.ascontiguousarray(B.conj().T if opB else B)
    tA, tB = torch.from_numpy(np.ascontiguousarray(A)).cuda(), torch.from_numpy(Bm).cuda()
    out = torch.full((A.shape[0], B.shape[1]), float("nan"), dtype=torch.complex128, device="cuda")
    assert lib.tebd_zgemm(precision, opB, A.shape[0], B.shape[1], A.shape[1], alpha, ctypes.c_void_p(tA.data_ptr()), A.shape[1],
                          ctypes.c_void_p(tB.data_ptr()), Bm.shape[1], ctypes.c_void_p(out.data_ptr()), B.shape[1],
                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    return out.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("opB", [0, 1])
@pytest.mark.parametrize("K", [1, 31, 130])  # 130: five k-steps, the row exponents by their own kernel
def test_exact_digits_bitwise(lib, opB, K):
    A, B = _rows(K, 0), _rows(K, 1).T
    ref = _digit_product(A, B)
    assert np.array_equal(_gpu(lib, 2, opB, A, B), ref)
    assert np.array_equal(_gpu(lib, 2, opB, A, B, -1.0), -ref)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf, 1e39])
def test_a_bad_value_stays_in_its_row(lib, precision, bad):
    r = np.random.Generator(np.random.PCG64(workloads.SEED))
    A = r.standard_normal((150, 70)) + 1j * r.standard_normal((150, 70))
    B = r.standard_normal((70, 90)) + 1j * r.standard_normal((70, 90))
    good = _gpu(lib, precision, 0, A, B)
    A2, B2 = A.copy(), B.copy()
    A2[41, 33] = bad
    B2[69, 64] = bad
    a, b = _gpu(lib, precision, 0, A2, B), _gpu(lib, precision, 0, A, B2)
    rows, cols = np.arange(150) != 41, np.arange(90) != 64
    assert np.array_equal(a[rows], good[rows]) and np.array_equal(b[:, cols], good[:, cols])
    if not (bad == 1e39 and precision != 1):
        assert not np.any(np.isfinite(a[41])) and not np.any(np.isfinite(b[:, 64]))
