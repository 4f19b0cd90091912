"""Calls when the device is nearly full."""
import ctypes

import numpy as np
import pytest

import workloads
from device_memory import MB, only

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opB", [0, 1])
@pytest.mark.parametrize("M,N,K", [(8192, 512, 2048), (1000, 4160, 2050)])
def test_split_tf32_product_in_blocks(lib, opB, M, N, K):
    """The operand planes of the whole product (300 MB) do not fit in what is left: the product runs block by
    block, with the same bits."""
    import torch
    A = torch.randn(M, K, dtype=torch.complex128, device="cuda")
    B = torch.randn(*((N, K) if opB else (K, N)), dtype=torch.complex128, device="cuda")
    ref, out = (torch.full((M, N), float("nan"), dtype=torch.complex128, device="cuda") for _ in range(2))

    def product(C):
        return lib.tebd_zgemm(1, opB, M, N, K, -0.75, ctypes.c_void_p(A.data_ptr()), K, ctypes.c_void_p(B.data_ptr()),
                              B.shape[1], ctypes.c_void_p(C.data_ptr()), N,
                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    assert product(ref) == 0
    with only(96 * MB):
        assert product(out) == 0
        torch.cuda.synchronize()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("form", ["dense", "supersite"])
def test_measurement_after_one_without_memory(lib, form):
    """A measurement whose buffers do not fit reports it; the next one, with memory, is the ordinary one."""
    from paper_2401_05301_gb300 import SuperSiteTEBD, TEBD
    from paper_2401_05301_gb300.binding import TEBDError
    args = (20, 3, 256, 4.0, 1.0, 0.1, 0.004, 10.5, 0.02) if form == "dense" else (20, 3, 128, 4.0, 1.0, 0.1, 0.004, 10.5, 0.02)

    def simulation():
        g = (TEBD if form == "dense" else SuperSiteTEBD)(*args)
        L, d = (20, 4) if form == "dense" else (10, 16)
        B, lam, _ = workloads.synthetic_state(L, d, args[2])
        g.set_state(B, lam)
        return g

    ref = simulation()
    n, cur = ref.measure()
    ref.close()
    g = simulation()
    with only(12 * MB):
        with pytest.raises(TEBDError) as e:
            g.measure()
        assert e.value.status == -2
    for a, b in zip(g.measure(), (n, cur)):
        assert np.array_equal(a, b)
    g.close()
