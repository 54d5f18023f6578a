"""GPU parity of the Hamiltonian step where its passes change: states smaller
than a tile, of one tile and of a few qubits more, more terms than a pass
takes, repeated pairs, one-body and diagonal terms only, real, imaginary and
general (non-Hermitian) entries, against the oracle."""
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


def terms_of(g, n, kind):
    X, Z = np.array([[0, 1], [1, 0]]), np.diag([1, -1])
    if kind == "diagonal":
        t = [([q], g.normal() * Z) for q in range(n)]
        return t + [([q, (q + 1) % n], np.kron(Z, Z) * g.normal()) for q in range(n - 1)]
    if kind == "field":
        return [([q], g.normal() * X) for q in range(n)]
    t = [([q], g.normal(size=(2, 2)) + 1j * g.normal(size=(2, 2))) for q in range(n)]
    for _ in range(3 * n if n > 1 else 0):
        a, b = (int(v) for v in g.permutation(n)[:2])
        t.append(([a, b], g.normal(size=(4, 4)) + 1j * g.normal(size=(4, 4))))
    return t


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("kind", ["general", "diagonal", "field"])
@pytest.mark.parametrize("n", [1, 2, 5, 11, 12, 13, 17])
def test_step_passes_vs_oracle(qc, n, kind, dt):
    g = W.rng(31 * n + dt)
    terms = terms_of(g, n, kind)
    v = W.random_state(g, n)
    s = qc.State(n, dt)
    s.load(v)
    x = v.astype(np.complex64).astype(np.complex128) if dt == 1 else v.copy()
    qc.qc_hamiltonian_step(s.h, 0.01, terms)
    O.hamiltonian_step(x, n, 0.01, terms)
    assert np.max(np.abs(s.numpy() - x)) <= (1e-12 if dt == 0 else 2e-5)
