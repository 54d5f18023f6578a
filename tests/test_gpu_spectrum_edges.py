"""GPU mixed-state spectrum at the edges of the eigenvalue solver: one to 64
universes around multiples of the cluster's rows, identical universes (rank
one), orthogonal ones (a diagonal Gram matrix, nothing to reduce), blocks of
repeated ones (repeated eigenvalues and exact zeros) and zero weights, against
numpy's eigenvalues of the oracle's rho."""
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


def batch(kind, g, n, B):
    N = 1 << n
    if kind == "random":
        v = g.normal(size=(B, N)) + 1j * g.normal(size=(B, N))
    elif kind == "same":
        v = np.tile(g.normal(size=N) + 1j * g.normal(size=N), (B, 1))
    elif kind == "orthogonal":
        v = np.zeros((B, N), dtype=complex)
        v[np.arange(B), g.permutation(N)[:B]] = np.exp(1j * g.random(B))
    else:  # blocks of repeated universes
        u = g.normal(size=(max(1, B // 4), N)) + 1j * g.normal(size=(max(1, B // 4), N))
        v = u[np.arange(B) % u.shape[0]]
    v = v / np.linalg.norm(v, axis=1, keepdims=True)
    P = g.random(B)
    if B > 2:
        P[1] = 0.0
    return v, P / P.sum()


@pytest.mark.parametrize("kind", ["random", "same", "orthogonal", "blocks"])
@pytest.mark.parametrize("B", [1, 2, 3, 7, 8, 9, 16, 33, 63, 64])
def test_spectrum_vs_numpy(qc, B, kind):
    import torch
    n = 7
    v, P = batch(kind, W.rng(B), n, B)
    psi = torch.tensor(v, dtype=torch.complex128, device="cuda")
    ev, (tr, p2, s) = qc.qc_mixed_spectrum(psi.data_ptr(), n, 0, B, P)
    w = v * np.sqrt(P)[:, None]
    ref = np.sort(np.linalg.eigvalsh(w.conj() @ w.T))[::-1]
    assert np.max(np.abs(ev - ref)) <= 1e-13
    assert abs(tr - 1) <= 1e-12 and abs(p2 - np.sum(ref ** 2)) <= 1e-12
    pos = ref[ref > 1e-14]
    assert abs(s + np.sum(pos * np.log(pos))) <= 1e-10
