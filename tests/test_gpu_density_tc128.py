"""GPU parity of the complex128 ensemble density matrix at the edges of its
tensor-core tiles: fewer amplitudes than a row or column block, one block and a
few, K chunks full and ragged, the largest batch of that path and the first of
the other, amplitudes over many orders of magnitude, and a NaN amplitude.
Each row is scaled to 55-bit integers and cut into seven 8-bit digits, and what
is dropped from a product is below 2^-51 of the two rows' largest entries: an
entry is within (2B 2^-54 + 2^-51) of the product of the rows' largest
magnitudes, plus binary64's own rounding of sqrt(P) C and of the result."""
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


def rho_gpu(qc, v, P):
    import torch
    B, N = v.shape
    psi = torch.tensor(v, dtype=torch.complex128, device="cuda")
    rho = torch.empty((N, N), dtype=torch.complex128, device="cuda")
    qc.qc_density_matrix(psi.data_ptr(), N.bit_length() - 1, 0, B, P, rho.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    return rho.cpu().numpy()


def states(g, n, B, spread):
    v = g.normal(size=(B, 1 << n)) + 1j * g.normal(size=(B, 1 << n))
    if spread:
        v *= 10.0 ** (-spread * g.random((B, 1 << n)))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


@pytest.mark.parametrize("spread", [0, 12])
@pytest.mark.parametrize("n,B", [(1, 1), (2, 3), (4, 8), (5, 64), (6, 7), (7, 9), (7, 64), (8, 16), (9, 33), (10, 64),
                                 (8, 65)])
def test_rho_vs_numpy(qc, n, B, spread):
    g = W.rng(10 * n + B)
    v = states(g, n, B, spread)
    P = g.random(B) + 0.1
    P /= P.sum()
    got = rho_gpu(qc, v, P)
    w = v * np.sqrt(P)[:, None]
    ref = w.T @ w.conj()
    top = np.max(np.maximum(np.abs(w.real), np.abs(w.imag)), axis=0)
    tol = (2 * B * 2.0 ** -54 + 2.0 ** -51 + 4 * B * 2.0 ** -53) * np.outer(top, top)
    if B <= 64:
        assert np.all(np.abs(got - ref) <= 2 * tol)  # real and imaginary parts, and numpy's own sums
        assert np.array_equal(got, got.conj().T)
        assert np.all(np.diag(got).imag == 0)
    else:  # CUDA cores, double-float
        assert np.max(np.abs(got - ref)) <= 1e-13


def test_rho_nan_amplitude(qc):
    g = W.rng(5)
    n, B = 8, 6
    v = states(g, n, B, 0)
    v[2, 77] = np.nan
    got = rho_gpu(qc, v, np.full(B, 1 / B))
    bad = np.zeros(1 << n, dtype=bool)
    bad[77] = True
    hit = bad[:, None] | bad[None, :]
    assert np.all(np.isnan(got[hit].real)) and np.all(np.isfinite(got[~hit]))
