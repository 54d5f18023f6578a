"""Calls of different sizes from two host threads, each on its own stream: a
kernel's limit of dynamic shared memory belongs to the device, so that a small
call must not take from a large one what it needs.  Every result equals the one
of the call alone."""
import threading

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


def gradient(qc, n, dt):
    import torch
    g = W.rng(n)
    gates = [(int(k), q, 0, 3 * q + int(k)) for q in range(n) for k in range(3)]
    gates += [(qc.QC_G_CNOT, q, (q + 1) % n, 0) for q in range(n)]
    c = qc.Circuit(n, gates, W.ansatz_hamiltonian(n), dt=dt)
    theta = torch.from_numpy(g.uniform(0, 6, (2, 3 * n))).cuda()
    return lambda: torch.cat([x.reshape(-1) for x in c.energy_and_grad(theta)])


def hamiltonian(qc, n, dt):
    import torch
    g = W.rng(n)
    m = g.normal(size=(n, 4, 4)) + 1j * g.normal(size=(n, 4, 4))
    terms = [([q, (q + 1) % n], m[q]) for q in range(n)]
    psi = torch.from_numpy(W.random_state(g, n)).cuda().to(torch.complex64 if dt else torch.complex128)

    def call():
        s = qc.State(n, dt, tensor=psi.clone())
        qc.qc_hamiltonian_step(s.h, 1e-2, terms)
        return s.tensor
    return call


def register_qft(qc, n, dt):
    import torch
    psi = torch.from_numpy(W.random_state(W.rng(n), n)).cuda().to(torch.complex64 if dt else torch.complex128)

    def call():
        s = qc.State(n, dt, tensor=psi.clone())
        qc.qc_qft_range(s.h, 1, n - 1)
        return s.tensor
    return call


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("make,small,large", [(register_qft, 4, 15), (gradient, 5, 16), (hamiltonian, 4, 14)])
def test_two_threads_of_different_size(qc, make, small, large, dt):
    import torch
    calls = [make(qc, n, dt) for n in (small, large)]
    want = [c() for c in calls]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                for _ in range(60):
                    got = calls[i]()
                    streams[i].synchronize()
                    assert torch.equal(got, want[i])
        except Exception as e:  # reported by the test's own thread
            errors.append((i, e))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
