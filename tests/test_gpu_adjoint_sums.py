"""GPU: the complex64 gradient's sums against complex128 of the same circuit:
few and many partial sums a thread, and observables far from 1 (the sums' point
follows the amplitudes)."""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0**-80, 1.0, 2.0**100])
@pytest.mark.parametrize("n", [2, 5, 9, 12, 13, 16])
def test_gradient_c64_vs_c128(n, scale):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_0902_0699_gb300 as qc
    g = W.rng(900 + n)
    gates, P = [], 0
    for layer in range(4):
        for q in range(n):
            gates += [(qc.QC_G_RY if (q + layer) % 3 else qc.QC_G_RX, q, 0, P), (qc.QC_G_RZ, q, 0, P + 1)]
            P += 2
        gates += [(qc.QC_G_CNOT, q, q + 1, 0) for q in range(n - 1)]
    terms = [(1, 0, 0.5), (0, 3, -0.7), (3, 1, 0.3), (1 << (n - 1), 1 << (n - 1), 0.2)]
    theta = g.random((4, P)) * 2 * math.pi
    grad = []
    for dt in (qc.QC_C128, qc.QC_C64):
        th = torch.tensor(theta, device="cuda", requires_grad=True)
        E = qc.energy(th, qc.Circuit(n, gates, [(x, z, c * scale) for x, z, c in terms], dt=dt))
        E.sum().backward()
        grad.append(th.grad.cpu().numpy() / scale)
    # three passes over len(gates) roundings of psi or lambda, each 2^-24 of its
    # norm at most and independent, times sum |c| = 1.7
    assert np.max(np.abs(grad[1] - grad[0])) <= 2.0**-24 * math.sqrt(3 * len(gates)) * 1.7
