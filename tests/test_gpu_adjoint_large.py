"""complex128 gradients of states whose backward sweep runs on thousands of
blocks with equal sums: the qubits above the tile are in equal superposition, so
that every tile holds the same amplitudes.  The state is a product, so the
gradient of sum_q c_q Z_q is -c_q sin theta_q."""
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


@pytest.mark.parametrize("n", [20, 26, 28])
def test_equal_tiles_closed_form(qc, n):
    import torch
    g = W.rng(n)
    low = 11
    th = g.uniform(0.3, 2.8, low)
    c = g.normal(size=low)
    gates = [(qc.QC_G_H, q, 0, 0) for q in range(low, n)] + [(qc.QC_G_RY, q, 0, q) for q in range(low)]
    terms = [(0, 1 << q, float(c[q])) for q in range(low)]
    circ = qc.Circuit(n, gates, terms)
    E, grad = circ.energy_and_grad(torch.from_numpy(th[None]).cuda())
    # two roundings of 2^-53 an operator and amplitude, n operators on psi and on lambda, relative to |H|
    tol = 4 * n * 2.0 ** -53 * np.abs(c).sum()
    assert abs(E.item() - np.dot(c, np.cos(th))) <= tol
    assert np.max(np.abs(grad[0].cpu().numpy() + c * np.sin(th))) <= tol
