"""GPU parity of parameterised circuits at the edges of the tile passes:
states smaller than a register block, of exactly one tile, and of one or two
qubits more, with all gate kinds, CNOTs between any two qubits and angles at
which a rotation's factor changes form (0, pi/2, pi, 2 pi), against the
oracle's gates and the parameter-shift rule."""
import math

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


def random_gates(g, n, count):
    """Gate list over all kinds; runs on one qubit and CNOT strings included."""
    gates, P = [], 0
    while len(gates) < count:
        q = int(g.integers(0, n))
        kind = int(g.integers(0, 6))
        if kind == 5:  # RY RZ on one qubit
            gates += [(1, q, 0, P), (2, q, 0, P + 1)]
            P += 2
        elif kind == 3:
            for _ in range(int(g.integers(1, 4))):
                c, t = (int(v) for v in g.permutation(n)[:2])
                gates.append((3, c, t, 0))
        elif kind == 4:
            gates.append((4, q, 0, 0))
        else:
            gates.append((kind, q, 0, P))
            P += 1
    return gates, P


def simulate(n, gates, theta):
    psi = O.zero_state(n)
    for kind, q0, q1, p in gates:
        if kind == 3:
            O.cnot(psi, n, q0, q1)
            continue
        if kind == 4:
            m = O.H_MAT
        elif kind == 0:
            c, s = math.cos(theta[p] / 2), math.sin(theta[p] / 2)
            m = np.array([[c, -1j * s], [-1j * s, c]])
        else:
            m = O.ry(theta[p]) if kind == 1 else O.rz(theta[p])
        O.apply_1q(psi, n, q0, m)
    return psi


def angles(g, P):
    th = g.random(P) * 2 * math.pi
    special = [0.0, math.pi / 2, math.pi, 2 * math.pi, -math.pi / 2, 1e-9]
    for k in range(0, P, 4):
        th[k] = special[(k // 4) % len(special)]
    return th


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n", [2, 3, 5, 10, 11, 12, 13, 14, 15])
def test_random_circuit_vs_oracle(qc, n, dt):
    import torch
    g = W.rng(100 * n + dt)
    gates, P = random_gates(g, n, 12 * n)
    B = 3
    theta = np.stack([angles(g, P) for _ in range(B)])
    th = torch.tensor(theta, device="cuda")
    psi = torch.empty(B << n, dtype=qc.torch_dtype(dt), device="cuda")
    qc.qc_circuit_forward(n, dt, B, gates, th.data_ptr(), P, psi.data_ptr())
    got = psi.cpu().numpy().reshape(B, -1)
    tol = 1e-12 if dt == 0 else 1e-5
    for b in range(B):
        assert np.max(np.abs(got[b] - simulate(n, gates, theta[b]))) <= tol


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n", [2, 4, 11, 12, 13, 14])
def test_gradient_vs_parameter_shift(qc, n, dt):
    import torch
    g = W.rng(200 * n + dt)
    gates, P = random_gates(g, n, 5 * n)
    terms = [(1, 0, 0.5), (0, 3, -0.7), (3, 1, 0.3), (1 << (n - 1), 1 << (n - 1), 0.2)]
    B = 2
    theta = np.stack([angles(g, P) for _ in range(B)])
    th = torch.tensor(theta, device="cuda", requires_grad=True)
    E = qc.energy(th, qc.Circuit(n, gates, terms, dt=dt))
    E.sum().backward()
    tol = 1e-12 if dt == 0 else 2e-5
    for b in range(B):
        assert abs(E[b].item() - O.energy(simulate(n, gates, theta[b]), n, terms)) <= tol
        for k in range(P):
            tp, tm = theta[b].copy(), theta[b].copy()
            tp[k] += math.pi / 2
            tm[k] -= math.pi / 2
            ps = 0.5 * (O.energy(simulate(n, gates, tp), n, terms) - O.energy(simulate(n, gates, tm), n, terms))
            assert abs(th.grad[b, k].item() - ps) <= tol


def test_unaligned_complex64_state(qc):
    """A complex64 batch needs 8-byte alignment only."""
    import torch
    n, B = 14, 2
    g = W.rng(9)
    gates, P = random_gates(g, n, 40)
    theta = np.stack([angles(g, P) for _ in range(B)])
    th = torch.tensor(theta, device="cuda")
    buf = torch.empty((B << n) + 1, dtype=torch.complex64, device="cuda")[1:]
    qc.qc_circuit_forward(n, 1, B, gates, th.data_ptr(), P, buf.data_ptr())
    ref = torch.empty(B << n, dtype=torch.complex64, device="cuda")
    qc.qc_circuit_forward(n, 1, B, gates, th.data_ptr(), P, ref.data_ptr())
    assert torch.equal(buf, ref)
