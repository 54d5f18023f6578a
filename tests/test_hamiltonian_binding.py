"""What the binding of the Hamiltonian step takes and refuses, and the term
records it hands to the library (no GPU, the library call is replaced)."""
import ctypes

import numpy as np
import pytest

import paper_0902_0699_gb300 as qc


@pytest.fixture()
def sent(monkeypatch):
    got = []

    class Lib:
        @staticmethod
        def qc_hamiltonian_step(h, dt, terms, n):
            p = ctypes.cast(terms, ctypes.POINTER(qc.HTerm))
            got.extend((p[i].k, list(p[i].qubits), np.array(p[i].h)) for i in range(n))
            return 0

    monkeypatch.setattr(qc, "lib", lambda: Lib)
    return got


@pytest.mark.parametrize("qubits", [[3], (3,), {3}, {3: "x"}.keys(), np.array([3], dtype=np.uint8), [np.int64(3)], range(3, 4),
                                    [3.0]])
def test_one_qubit_terms(sent, qubits):
    m = np.array([[1, 2j], [-2j, 0.5]])
    qc.qc_hamiltonian_step(None, 0.1, [(qubits, m)])
    k, q, h = sent[0]
    assert k == 1 and q == [3, 0]
    assert np.array_equal(h[:8], [1, 0, 0, 2, 0, -2, 0.5, 0]) and not h[8:].any()


@pytest.mark.parametrize("form", [list, np.asfortranarray, lambda m: m.real, lambda m: m[::-1][::-1]])
def test_two_qubit_matrices(sent, form):
    m = np.arange(16).reshape(4, 4) * (1 + 1j)
    qc.qc_hamiltonian_step(None, 0.1, [([0, 1], np.eye(4)), ([5, 2], form(m))])
    k, q, h = sent[1]
    want = np.asarray(form(m), dtype=complex).reshape(-1)
    assert k == 2 and q == [5, 2] and np.array_equal(h[0::2], want.real) and np.array_equal(h[1::2], want.imag)


@pytest.mark.parametrize("term", [([0, 1, 2], np.eye(4)), ([0, 1], np.eye(8))])
def test_too_large(sent, term):
    with pytest.raises(IndexError):
        qc.qc_hamiltonian_step(None, 0.1, [term])
    assert not sent
