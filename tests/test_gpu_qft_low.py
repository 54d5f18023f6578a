"""The register QFT near the bottom of the state, where a tile is filled by
index bits above the register, and on one qubit: against numpy, and with columns
of very different size (complex128)."""
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


CASES = [(n, lo, w) for n in (5, 11, 12, 13, 14, 16) for lo in (0, 1, 3) for w in (1, 2, 3, 5, 8, 10) if lo + w <= n]
CASES += [(16, 1, 12), (17, 1, 13), (16, 2, 13), (17, 0, 12)]


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,lo,w", CASES)
def test_low_register(qc, n, lo, w, dt):
    g = W.rng(1000 * n + 10 * lo + w)
    v = W.random_state(g, n).reshape(-1, 1 << w, 1 << lo)
    if dt == 0:
        v = v * 10.0 ** (-20 * g.random((v.shape[0], 1, v.shape[2])))
    else:
        v = v.astype(np.complex64).astype(np.complex128)
    s = qc.State(n, dt)
    s.load(v.reshape(-1))
    qc.qc_qft_range(s.h, lo, w)
    got = s.numpy().astype(np.complex128).reshape(v.shape)
    ref = np.fft.ifft(v, axis=1, norm="ortho")
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    # complex128: six roundings a pass to 2^-54 of a column's largest amplitude, at most
    # 2^(k/2) of its norm; complex64: a rounding of each factor, product and sum of a level
    assert np.max(err) <= (2.0 ** -44 if dt == 0 else 4 * w * 2.0 ** -24)
