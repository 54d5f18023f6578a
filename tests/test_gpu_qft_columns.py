"""The register QFT transforms the columns of its tiles independently: for every
value of the qubits outside the register.  Columns far below their neighbours
keep their accuracy, subnormal ones included, and an infinity or a NaN stays in
its own column."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = [(6, 2, 3), (8, 5, 1), (10, 7, 2), (12, 3, 6), (12, 1, 11), (13, 11, 2), (16, 4, 12), (17, 6, 11)]


@pytest.fixture(scope="module")
def qc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_0902_0699_gb300 as q
    q.lib()
    return q


def run(qc, v, n, lo, w):
    s = qc.State(n, 0)
    s.load(v)
    qc.qc_qft_range(s.h, lo, w)
    return s.numpy().reshape(1 << (n - lo - w), 1 << w, 1 << lo)


def dft(v, n, lo, w):
    t = v.reshape(1 << (n - lo - w), 1 << w, 1 << lo)
    return np.fft.ifft(t, axis=1, norm="ortho")


@pytest.mark.parametrize("n,lo,w", CASES)
def test_columns_of_different_size(qc, n, lo, w):
    g = W.rng(100 * n + w)
    v = W.random_state(g, n).reshape(-1, 1 << w, 1 << lo)
    v = v * 10.0 ** (-30 * g.random((v.shape[0], 1, v.shape[2])))
    got, ref = run(qc, v.reshape(-1), n, lo, w), dft(v, n, lo, w)
    # an amplitude has 54 bits or more below its column's largest, and a pass of k levels rounds
    # (k + 1) / 2 times: 2^(k/2) k 2^-54 of a column's norm at most, for two passes of six levels
    # or one of eleven below 2^-44
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.max(err) <= 2.0 ** -44


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n,lo,w", CASES)
def test_not_finite_stays_in_its_column(qc, n, lo, w, bad):
    g = W.rng(n)
    v = W.random_state(g, n)
    ref = dft(v, n, lo, w)
    at = int(g.integers(0, 1 << n))
    v[at] = bad
    got = run(qc, v, n, lo, w)
    hit = np.zeros(1 << n, dtype=bool)
    hit[at] = True
    col = np.zeros(got.shape, dtype=bool) | hit.reshape(got.shape).any(axis=1, keepdims=True)
    assert not np.any(np.isfinite(got[col]))
    assert np.max(np.abs(got[~col] - ref[~col])) <= 2.0 ** -44


@pytest.mark.parametrize("n,lo,w", CASES)
def test_subnormal_columns(qc, n, lo, w):
    g = W.rng(n + w)
    v = W.random_state(g, n).reshape(-1, 1 << w, 1 << lo)
    tiny = g.random((v.shape[0], 1, v.shape[2])) < 0.5
    tiny[0, 0, 0] = True
    unit = 2.0 ** -1074
    v = np.where(tiny, np.ldexp(np.rint(v.real * 2.0 ** 45), -1074) + 1j * np.ldexp(np.rint(v.imag * 2.0 ** 45), -1074), v)
    got, big = run(qc, v.reshape(-1), n, lo, w), dft(v * 2.0 ** 1000, n, lo, w) * 2.0 ** -1000
    col = np.broadcast_to(tiny, got.shape)
    # fixed point in 2^-1076 or finer, rounded (k + 1) / 2 times a pass; numpy's own rounding, half a unit each
    d = (got - big)[col]
    assert np.max(np.abs(d.real)) <= 4 * unit * (1 + w // 6) and np.max(np.abs(d.imag)) <= 4 * unit * (1 + w // 6)
    assert np.any(got[col] != 0)
