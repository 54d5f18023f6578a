"""Seeded sampling with more shots than blocks (sums of 32 weights) at block
edges, against the oracle's outcomes, and the library's workspace pool: calls
interleaved on two streams and from two threads give what they give alone, also
after every handle was freed."""
import threading

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
@pytest.mark.parametrize("n,shots,kind", [(1, 40, "random"), (4, 100, "random"), (5, 100, "random"), (6, 300, "peak"),
                                          (11, 50, "random"), (12, 3000, "zeros"), (13, 4000, "random"),
                                          (17, 5000, "peak"), (18, 9000, "random")])
def test_many_shots_vs_oracle(qc, n, shots, kind, dt):
    g = W.rng(n + shots)
    v = W.random_state(g, n)
    if kind == "peak":  # nearly all weight on the last amplitude
        v *= 1e-4
        v[-1] = 1
    elif kind == "zeros":  # whole runs of 32 and whole blocks without weight
        v[: 1 << (n - 1)] = 0
        v[np.arange(1 << n) % 64 < 40] = 0
    s = qc.State(n, dt)
    s.load(v / np.linalg.norm(v))
    w = s.numpy().astype(np.complex128)
    p = w.real * w.real + w.imag * w.imag
    ref = O.sample_from_probs(p, 11, shots)
    assert np.array_equal(s.sample(11, shots).cpu().numpy().astype(np.uint64), ref)
    pg, got = s.probs_sample(11, shots)
    assert np.array_equal(got.cpu().numpy().astype(np.uint64), ref)
    assert np.array_equal(pg.cpu().numpy(), p)


def run_on(qc, stream, n, seed, out):
    import torch
    with torch.cuda.stream(stream):
        t = torch.from_numpy(W.random_state(W.rng(seed), n)).cuda()
        s = qc.State(n, 0, tensor=t)
        for _ in range(5):
            s.qft()
            s.sample(seed, 2000)
        out[seed] = s.tensor.clone()
        s.close()


def test_pool_two_streams_and_threads(qc):
    import torch
    n = 15
    alone, both, threads = {}, {}, {}
    for seed in (1, 2):
        run_on(qc, torch.cuda.current_stream(), n, seed, alone)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for seed, st in ((1, a), (2, b)):
        run_on(qc, st, n, seed, both)
    ts = [threading.Thread(target=run_on, args=(qc, st, n, seed, threads)) for seed, st in ((1, a), (2, b))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for seed in (1, 2):
        assert torch.equal(alone[seed], both[seed]) and torch.equal(alone[seed], threads[seed])
