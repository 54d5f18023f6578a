"""The sampler on both sides of the rule that takes the full CDF (2^14 shots and
a 32nd of the amplitudes), at the smallest states and block edges, against the
oracle's outcomes."""
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
@pytest.mark.parametrize("n,shots", [(1, 16384), (5, 16383), (5, 40000), (11, 16384), (12, 30000), (18, 16384), (19, 16383),
                                     (19, 16384), (20, 16384), (20, 32768)])
def test_outcomes_vs_oracle(qc, n, shots, dt):
    v = W.random_state(W.rng(n + shots), n)
    v[np.arange(1 << n) % 7 == 3] = 0
    s = qc.State(n, dt)
    s.load(v / np.linalg.norm(v))
    w = s.numpy().astype(np.complex128)
    p = w.real * w.real + w.imag * w.imag
    ref = O.sample_from_probs(p, 11, shots)
    assert np.array_equal(s.sample(11, shots).cpu().numpy().astype(np.uint64), ref)
    pg, got = s.probs_sample(11, shots)
    assert np.array_equal(got.cpu().numpy().astype(np.uint64), ref)
    assert np.array_equal(pg.cpu().numpy(), p)
