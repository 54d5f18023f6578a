"""GPU parity of the one-block Grover run over its whole range of sizes and
marked counts (warp edges, everything marked, zero to many iterations) against
the oracle's literal operators, and its accuracy against the closed form."""
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


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,m,iters", [(1, 1, 3), (2, 3, 5), (2, 4, 2), (3, 2, 0), (5, 32, 4), (6, 17, 9), (7, 33, 5),
                                       (9, 5, 17), (10, 1, 25), (11, 1024, 7), (12, 64, 6), (13, 3, 41), (13, 1000, 3)])
def test_run_vs_oracle(qc, n, m, iters, dt):
    marked = W.marked_indices(W.rng(n + m), n, m)
    s = qc.State(n, dt)
    s.grover_run(marked, iters)
    ref = O.zero_state(n)
    O.hall(ref, n)
    for _ in range(iters):
        O.grover_step(ref, n, marked)
    assert np.max(np.abs(s.numpy() - ref)) <= (1e-12 if dt == 0 else 1e-6)


@pytest.mark.parametrize("n,m", [(10, 1), (13, 4)])
def test_run_closed_form(qc, n, m):
    marked = W.marked_indices(W.rng(3 * n), n, m)
    k, N = W.grover_iterations(n), 1 << n
    s = qc.State(n, 0)
    s.grover_run(marked, k)
    t = math.asin(math.sqrt(m / N))
    ref = np.full(N, math.cos((2 * k + 1) * t) / math.sqrt(N - m))
    ref[marked.astype(int)] = math.sin((2 * k + 1) * t) / math.sqrt(m)
    # the step's only rounding is 2^-63; the closed form itself is good to k ulps
    assert np.linalg.norm(s.numpy() - ref) <= 1e-14
