"""complex128 density matrices whose entries are far below the product of their
rows' largest magnitudes: universes near different basis states that leak a
little into the others, some of them disjoint, beside ordinary ones.  An entry
has to be good to its own terms sum_a P_a |C_a(i)| |C_a(j)|, which double-float
products keep to about 2^-47."""
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
    rho = torch.full((N, N), 7.0 + 7.0j, dtype=torch.complex128, device="cuda")
    qc.qc_density_matrix(psi.data_ptr(), N.bit_length() - 1, 0, B, P, rho.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    return rho.cpu().numpy()


def leaky(g, n, B, leak, kind):
    N = 1 << n
    v = leak * (g.normal(size=(B, N)) + 1j * g.normal(size=(B, N)))
    if kind == "disjoint":  # exact zeros: every state has its own amplitudes only
        v[np.arange(B)[:, None] != np.arange(N)[None, :] % B] = 0
    own = g.integers(0, N, B) if kind == "few" else None
    if own is not None:
        v[np.arange(B), own] = 1
    else:  # state a is large where i = a mod B
        big = np.arange(B)[:, None] == np.arange(N)[None, :] % B
        v[big] += g.normal(size=big.sum())
    if kind == "mixed" and N >= 256:  # ordinary amplitudes in the second half
        v[:, N // 2:] = g.normal(size=(B, N // 2)) + 1j * g.normal(size=(B, N // 2))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


@pytest.mark.parametrize("kind", ["own", "few", "disjoint", "mixed"])
@pytest.mark.parametrize("leak", [1e-4, 1e-16])
@pytest.mark.parametrize("n,B", [(1, 2), (3, 3), (6, 7), (7, 64), (8, 2), (9, 33), (10, 64)])
def test_entries_to_their_own_terms(qc, n, B, leak, kind):
    g = W.rng(100 * n + B)
    v = leaky(g, n, B, leak, kind)
    P = g.random(B) + 0.1
    P /= P.sum()
    got = rho_gpu(qc, v, P)
    w = v * np.sqrt(P)[:, None]
    ref = w.T @ w.conj()
    size = np.abs(w).T @ np.abs(w)
    # double-float products and sums: a few 2^-47 a term; digits: 2^-49.4 of the
    # scales' product a real product, where that is at most 26 / sqrt(2 B) of the
    # terms; numpy's own sums; 1e-33: what a float pair keeps of an amplitude
    # below 2^-74
    tol = (2.0 ** -44 + 2 * B * 2.0 ** -49.4 * 26 / np.sqrt(2 * B) + 4 * B * 2.0 ** -53) * size + 1e-33
    err = np.abs(got - ref)
    assert np.all(err <= tol), np.max(err / tol)
    assert np.array_equal(got, got.conj().T)
    assert np.all(np.diag(got).imag == 0)
