"""complex128 circuits where the forward sweep's tiles change size with the
number of tiles (qubits and batch), with passes of one RZ, of two and of none,
against the gates applied one by one."""
import ctypes

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


def circuit(g, n, kind):
    """(kind, q0, q1, param) over RX, RY, RZ, CNOT and H."""
    ops = []
    if kind == "one RZ":  # alone, behind operators, behind a CNOT
        ops = [(4, 0, 0), (1, n - 1, 0), (3, n - 1, 0), (2, 0, 0), (3, 0, n - 1), (2, n // 2, 0)]
    else:
        for _ in range(40 if kind == "mixed" else 12):
            a, b = (int(v) for v in g.permutation(n)[:2])
            k = int(g.integers(0, 5))
            ops.append((k, a, b if k == 3 else 0))
        if kind == "no rotation":
            ops = [(4 if k != 3 else 3, a, b) for k, a, b in ops]
    gates, p = [], 0
    for k, a, b in ops:
        gates.append((k, a, b, p if k <= 2 else 0))
        p += k <= 2
    return gates, p


@pytest.mark.parametrize("kind", ["one RZ", "mixed", "no rotation"])
@pytest.mark.parametrize("n,B", [(2, 1), (9, 1), (10, 1), (11, 1), (12, 1), (14, 1), (19, 1), (20, 1), (11, 64), (12, 16),
                                 (13, 64), (14, 3)])
def test_forward_vs_gates(qc, n, B, kind):
    import torch
    g = W.rng(n * 100 + B)
    gates, P = circuit(g, n, kind)
    c = qc.Circuit(n, gates, [(0, 1, 1.0)])
    theta = torch.from_numpy(g.uniform(0, 6, (B, max(P, 1)))).cuda()
    psi = torch.empty(B << n, dtype=torch.complex128, device="cuda")
    V = ctypes.c_void_p
    assert qc.lib().qc_circuit_forward(n, 0, B, c.gates, c.n_gates, V(theta.data_ptr()), theta.shape[1],
                                       V(psi.data_ptr()), V(torch.cuda.current_stream().cuda_stream)) == 0
    for b in sorted({0, B // 2, B - 1}):
        s = qc.State(n, 0)
        s.reset(0)
        t = theta[b].cpu().numpy()
        for k, a, q1, p in gates:
            if k == 3:
                s.cnot(a, q1)
                continue
            x, y = np.cos(t[p] / 2), np.sin(t[p] / 2)
            h = np.sqrt(0.5)
            m = {0: [[x, -1j * y], [-1j * y, x]], 1: [[x, -y], [y, x]], 2: [[x - 1j * y, 0], [0, x + 1j * y]],
                 4: [[h, h], [h, -h]]}[k]
            s.apply_1q(a, np.array(m, dtype=complex))
        assert torch.max(torch.abs(psi[b << n:(b + 1) << n] - s.tensor)).item() <= 1e-13
