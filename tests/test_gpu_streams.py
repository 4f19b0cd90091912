"""A handle on a non-blocking stream, which does not wait for the legacy stream that uploads run on."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
def test_step_at_once_on_a_non_blocking_stream(lib, order):
    """Gates, state and step follow one another without a wait by the caller; the result is that of the default
    stream, bitwise."""
    import torch
    from paper_2401_05301_gb300 import TEBD
    L, d, chi = 12, 4, 96
    B, lam, _ = workloads.synthetic_state(L, d, chi)

    def run(stream):
        g = TEBD(L, d - 1, chi, 4.0, 1.0, 0.1, 0.004, 6.5, 0.02)
        if stream is not None:
            g.set_stream(stream.cuda_stream)
        g.set_option("trotter_order", order)
        g.set_state(B, lam)
        g.step(1)
        out = g.measure()
        g.close()
        return out

    ref = run(None)
    for _ in range(3):
        for a, b in zip(run(torch.cuda.Stream()), ref):
            assert np.array_equal(a, b)
