"""Small Grover runs where the marked amplitudes' sum changes form: four warps of
partial sums, five, a last one of a single item, and all thirty-two."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,m", [(8, 128), (8, 129), (9, 160), (9, 161), (10, 512), (10, 1000), (13, 129), (13, 1024)])
def test_many_marked_vs_oracle(n, m, dt):
    import paper_0902_0699_gb300 as qc
    marked = W.marked_indices(W.rng(n + m), n, m)
    s = qc.State(n, dt)
    s.grover_run(marked, 6)
    ref = O.zero_state(n)
    O.hall(ref, n)
    for _ in range(6):
        O.grover_step(ref, n, marked)
    assert np.max(np.abs(s.numpy() - ref)) <= (1e-12 if dt == 0 else 1e-6)
