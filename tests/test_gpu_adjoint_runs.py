"""complex64 derivative sums of long runs of rotations on the same qubits (one
register round of up to forty operators).  The run's angles are zero, so that
its operators change no amplitude, and H is one Pauli string: the derivatives
are then Im <H psi|P|psi> of the complex64 state itself, with no rounding but
that of the sums."""
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


def pauli(v, x, z):
    j = np.arange(v.size)
    sign = 1 - 2 * np.array([bin(int(k)).count("1") & 1 for k in (j ^ x) & z])
    return 1j ** bin(x & z).count("1") * sign * v[j ^ x]


@pytest.mark.parametrize("per", [2, 5, 13])
@pytest.mark.parametrize("n", [6, 14])
def test_run_of_rotations(qc, n, per):
    import ctypes
    import torch
    g = W.rng(n)
    gates = [(k, q, 0, 2 * q + k - 1) for q in range(n) for k in (1, 2)]  # RY, RZ on every qubit
    gates += [(qc.QC_G_CNOT, q, (q + 1) % n, 0) for q in range(n)]
    P0 = 2 * n
    run = [(int(g.integers(0, 3)), q) for _ in range(per) for q in range(3)]
    gates += [(k, q, 0, P0 + i) for i, (k, q) in enumerate(run)]
    theta = np.zeros(P0 + len(run))
    theta[:P0] = g.uniform(0, 6, P0)
    x, z = 0b000011, 0b001010  # X0 Y1 Z3
    circ = qc.Circuit(n, gates, [(x, z, 1.0)], dt=1)
    th = torch.from_numpy(theta[None]).cuda()
    _, grad = circ.energy_and_grad(th)
    psi = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    V = ctypes.c_void_p
    assert qc.lib().qc_circuit_forward(n, 1, 1, circ.gates, circ.n_gates, V(th.data_ptr()), theta.size,
                                       V(psi.data_ptr()), V(torch.cuda.current_stream().cuda_stream)) == 0
    v = psi.cpu().numpy().astype(np.complex128)
    lam = pauli(v, x, z)
    want = [np.vdot(lam, pauli(v, [1 << q, 1 << q, 0][k], [0, 1 << q, 1 << q][k])).imag for k, q in run]
    # 16 products a thread and operator, each to 2^-24 of a unit of 2^-13 of the largest products
    tol = 16 * 2.0 ** -37 * (1 << (n - 3)) * np.max(np.abs(v)) ** 2
    got = grad[0, P0:].cpu().numpy()
    assert np.max(np.abs(got - want)) <= tol, (np.max(np.abs(got - want)), tol)
