"""GPU parity of the register QFT at the edges of its passes: single-pass
registers with rows of one to many amplitudes, the first sizes that take two
groups and a reversal pass, registers at the bottom and the top of the state;
and projections onto single amplitudes and whole registers."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_0902_0699_gb300 as q
    q.lib()
    return q


CASES = [(1, 0, 1), (2, 1, 1), (3, 0, 2), (6, 2, 3), (9, 0, 5), (12, 1, 11), (13, 2, 11), (13, 1, 12), (14, 0, 13),
         (15, 3, 12), (15, 0, 12), (16, 1, 14), (17, 6, 11), (18, 0, 17), (18, 4, 9), (19, 9, 10), (20, 1, 19)]


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,lo,w", CASES)
def test_register_qft_vs_oracle(qc, n, lo, w, dt):
    v = W.random_state(W.rng(1000 * n + 10 * lo + w), n)
    s = qc.State(n, dt)
    s.load(v)
    qc.qc_qft_range(s.h, lo, w)
    x = v.astype(np.complex64).astype(np.complex128) if dt else v.copy()
    O.qft_range(x, n, lo, w)
    assert np.max(np.abs(s.numpy() - x)) <= (1e-12 if dt == 0 else 1e-5)


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,lo,w", [(1, 0, 1), (6, 0, 6), (9, 0, 3), (9, 6, 3), (12, 5, 2), (14, 1, 12)])
def test_projection_vs_oracle(qc, n, lo, w, dt):
    g = W.rng(77 * n + lo)
    v = W.random_state(g, n)
    value = int(g.integers(0, 1 << w))
    s = qc.State(n, dt)
    s.load(v)
    p = qc.qc_project(s.h, lo, w, value)
    x = v.astype(np.complex64).astype(np.complex128) if dt else v.copy()
    keep = ((np.arange(1 << n) >> lo) & ((1 << w) - 1)) == value
    pr = float(np.sum(np.abs(x[keep]) ** 2))
    x = np.where(keep, x, 0) / np.sqrt(pr)
    assert abs(p - pr) <= 1e-12
    got = s.numpy()
    assert np.max(np.abs(got - x)) <= (1e-12 if dt == 0 else 1e-5)
    assert np.all(got[~keep] == 0)
