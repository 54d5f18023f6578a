"""GPU parity of the complex64 QFT at the edges of its passes: the largest
single tile (12 qubits), the first sizes of the bit reversal's kernel with a
group of eight, nine and ten levels above it, two groups and three."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [11, 12, 13, 14, 15, 16, 21, 22, 24])
def test_qft_c64_error_in_two_norm(n):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_0902_0699_gb300 as qc
    v = W.random_state(W.rng(300 + n), n).astype(np.complex64).astype(np.complex128)
    s = qc.State(n, qc.QC_C64)
    s.load(v)
    s.qft()
    ref = O.qft(v.copy(), n)
    # a level rounds an addition and a product, each group a twiddle: about
    # 4 n independent roundings of 2^-24 per amplitude
    assert np.linalg.norm(s.numpy() - ref) <= 2.0**-24 * np.sqrt(4 * n) * np.linalg.norm(ref)
    s.close()
