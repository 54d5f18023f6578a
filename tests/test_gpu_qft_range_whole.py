"""The complex128 register QFT on a register that is the whole state keeps the
accuracy of a smaller register's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_0902_0699_gb300 as q
    q.lib()
    return q


@pytest.mark.parametrize("n", [1, 4, 8, 11, 12, 13, 17, 20, 21, 23])
def test_whole_state_register(qc, n):
    v = W.random_state(W.rng(n), n)
    s = qc.State(n, 0)
    s.load(v)
    qc.qc_qft_range(s.h, 0, n)
    ref = np.fft.ifft(v, norm="ortho")
    # a pass rounds at most six times to 2^-54 of the largest amplitude, which is within eight
    # times the root mean square; numpy's transform: 2^-53 a level or less
    passes = 1 if n <= 11 else 2 if n <= 20 else 3
    tol = passes * 6 * 2.0 ** -51 + 2.0 ** -53 * np.sqrt(n)
    assert np.linalg.norm(s.numpy() - ref) <= tol
