"""What the performance of this library is measured on.

Twelve listed cases, one for each kind of program the library serves, and
`draw` for more of the same ranges: the smallest calls (a 10-qubit search, a
17-qubit period finding) up to a 30-qubit complex128 state, complex128 and
complex64, forward and gradient.  Every pass goes through the public entry
points of paper_0902_0699_gb300 and returns the state, matrix or gradient the
call computes.

A case is a dict with its "family" and sizes; "dt" is 0 for complex128 and 1
for complex64.  Quantities that the library derives in FP64 from a complex64
state which a case has just computed (probabilities, samples) are returned
for complex128 only: there they are functions of the state to FP64 accuracy.
"""
import math

import numpy as np
import torch

import paper_0902_0699_gb300 as qc
import workloads as W

C128, C64 = qc.QC_C128, qc.QC_C64


def listed():
    return [
        # sec. 5.1's textbook search: a small state, one call and a read-out;
        # what counts is the latency of the calls
        dict(name="grover_n10", family="search", n=10, dt=C128, marked=1, iters=25, shots=100),
        # period finding for M = 33 (11 + 6 qubits): preparation, projective
        # measurement, register QFT, read-out on a state that fits the L2 cache
        dict(name="shor_m33", family="shor", M=33, dt=C128, shots=1000),
        # the headline program at its size: Grover operators on 2^30
        # amplitudes, the QFT, probabilities and 1000 samples
        dict(name="grover_qft_n30_c128", family="grover_qft", n=30, dt=C128, marked=8, iters=10, shots=1000),
        # the complex64 QFT on a large state with an odd qubit count
        dict(name="qft_n29_c64", family="qft", n=29, dt=C64),
        # a layer of a random circuit, gate by gate: a Haar U(2) on every qubit
        # and a brick wall of CNOTs
        dict(name="circuit_n24_c128", family="circuit", n=24, dt=C128, layers=1),
        # ten layers of the same circuit in complex64, fused into dense blocks
        # once and then run
        dict(name="fused_n24_c64", family="fused", n=24, dt=C64, layers=10),
        # variational training, single precision: energies and gradients of a
        # batch of 64 angle sets of a 20-qubit ansatz
        dict(name="adjoint_n20_b64_c64", family="adjoint", n=20, dt=C64, batch=64, layers=10),
        # the same gradient for one angle set in double precision
        dict(name="adjoint_n20_b1_c128", family="adjoint", n=20, dt=C128, batch=1, layers=10),
        # noisy trajectories of uneven sizes (sec. 6.2-6.3), one launch
        dict(name="traj_512", family="traj", inst=512, n_lo=12, n_hi=18, p=1e-3),
        # the ensemble density matrix and its spectrum (sec. 6.1)
        dict(name="rho_n13_b64_c128", family="rho", n=13, dt=C128, batch=64),
        # two first-order steps under a Heisenberg chain in a field (sec. 7)
        dict(name="hamiltonian_n22_c128", family="hamiltonian", n=22, dt=C128, steps=2),
        # observables and read-out of a stored complex64 state: normalisation,
        # Pauli strings, probabilities and more shots than blocks
        dict(name="measure_n26_c64", family="measure", n=26, dt=C64, terms=8, shots=100000),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the listed families, over their whole ranges."""
    f = rng.choice(["search", "shor", "grover_qft", "qft", "circuit", "fused", "adjoint", "adjoint", "traj", "rho",
                    "hamiltonian", "measure"])
    dt = rng.choice([C128, C64])
    if f == "search":
        n = rng.randint(6, 13)
        return dict(family=f, n=n, dt=dt, marked=rng.randint(1, 4), iters=rng.randint(1, W.grover_iterations(n)),
                    shots=_log_int(rng, 1, 2000))
    if f == "shor":
        return dict(family=f, M=_log_int(rng, 15, 380), dt=dt, shots=_log_int(rng, 10, 4000))
    if f == "grover_qft":
        return dict(family=f, n=rng.randint(12, 28), dt=dt, marked=_log_int(rng, 1, 64), iters=rng.randint(1, 12),
                    shots=_log_int(rng, 1, 5000))
    if f == "qft":
        return dict(family=f, n=rng.randint(6, 28), dt=dt)
    if f == "circuit":
        return dict(family=f, n=rng.randint(6, 26), dt=dt, layers=rng.randint(1, 2))
    if f == "fused":
        return dict(family=f, n=rng.randint(8, 25), dt=dt, layers=rng.randint(2, 10))
    if f == "adjoint":
        n = rng.randint(6, 20)
        most = max(1, min(64, 1 << ((25 if dt == C64 else 23) - n)))
        return dict(family=f, n=n, dt=dt, batch=_log_int(rng, 1, most), layers=rng.randint(2, 10 if dt == C64 else 6))
    if f == "traj":
        lo = rng.randint(6, 14)
        return dict(family=f, inst=_log_int(rng, 8, 512), n_lo=lo, n_hi=rng.randint(lo, 17),
                    p=rng.choice([1e-4, 1e-3, 4e-3]))
    if f == "rho":
        return dict(family=f, n=rng.randint(5, 13), dt=dt, batch=rng.randint(2, 64))
    if f == "hamiltonian":
        return dict(family=f, n=rng.randint(6, 24), dt=dt, steps=rng.randint(1, 3))
    return dict(family=f, n=rng.randint(8, 27), dt=dt, terms=rng.randint(2, 10), shots=_log_int(rng, 10, 200000))


# ------------------------------------------------------------------ inputs --

def _rng(seed):
    return W.rng(seed & 0x7FFFFFFF)


def _state(n, seed, dt, batch=None):
    """Gaussian amplitudes, each state normalised (complex128 until the end,
    so that both types hold the same state)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = 1 if batch is None else batch
    v = torch.randn((rows, 2 << n), generator=g, device="cuda", dtype=torch.float32 if dt == C64 else torch.float64)
    v.div_(v.norm(dim=1, keepdim=True))
    v = torch.view_as_complex(v.view(rows, 1 << n, 2))
    return v[0].contiguous() if batch is None else v


def _circuit(case, seed):
    g = _rng(seed + 1)
    n = case["n"]
    return [(W.haar_u2(g, n), [(i, i + 1) for i in range(l % 2, n - 1, 2)]) for l in range(case["layers"])]


def _ansatz(case):
    """The layered ansatz RY, RZ on every qubit and a CNOT ring, and
    H = Z0 Z1 + 0.1 sum X_i, as gate and Pauli lists."""
    n, gates = case["n"], []
    for l in range(case["layers"]):
        for q in range(n):
            gates.append((qc.QC_G_RY, q, 0, l * 2 * n + 2 * q))
            gates.append((qc.QC_G_RZ, q, 0, l * 2 * n + 2 * q + 1))
        for q in range(n):
            gates.append((qc.QC_G_CNOT, q, (q + 1) % n, 0))
    return gates, W.ansatz_hamiltonian(n)


def _theta(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.rand((case["batch"], case["layers"] * 2 * case["n"]), generator=g, device="cuda", dtype=torch.float64)
    return (t * 2 * math.pi).to(torch.float64 if case["dt"] == C128 else torch.float32)


def _shor(case, seed):
    M = case["M"]
    n2 = max(1, math.ceil(math.log2(M)))
    n1 = math.ceil(math.log2(M * M))
    xs = [x for x in range(2, M) if math.gcd(x, M) == 1]
    return n1, n2, xs[seed % len(xs)]


def _chain(case, seed):
    """A Heisenberg chain with seeded couplings in a seeded field."""
    g = _rng(seed + 2)
    X, Y, Z = np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])
    xx, yy, zz = np.kron(X, X), np.kron(Y, Y), np.kron(Z, Z)
    n = case["n"]
    terms = [([q], g.normal() * X + g.normal() * Z) for q in range(n)]
    terms += [([q, q + 1], g.normal() * xx + g.normal() * yy + g.normal() * zz) for q in range(n - 1)]
    return terms


def _strings(case, seed):
    """Pauli strings of one to three factors, Z-only ones among them."""
    g = _rng(seed + 3)
    out = []
    for k in range(case["terms"]):
        x = z = 0
        for q in g.permutation(case["n"])[:1 + k % 3]:
            kind = 2 if k % 2 else int(g.integers(0, 3))
            x |= int(kind != 2) << int(q)
            z |= int(kind != 0) << int(q)
        out.append((x, z))
    return out


def _ensemble(case, seed):
    """Universes that share a large part of one state and differ by noise."""
    v = _state(case["n"], seed, case["dt"], case["batch"])
    v = v + 1.5 * v[:1]
    v = (v / v.abs().pow(2).sum(dim=1, keepdim=True).sqrt()).contiguous()
    P = _rng(seed + 4).random(case["batch"]) + 0.1
    return v, P / P.sum()


def _fused_ops(case, seed):
    ops = []
    for U, pairs in _circuit(case, seed):
        ops += [(qc.QC_OP_1Q, q, 0, 0, U[q]) for q in range(case["n"])]
        ops += [(qc.QC_OP_CNOT, c, t, 0, None) for c, t in pairs]
    return ops


def prepare(case, seed):
    f, st = case["family"], {"case": case, "seed": seed}
    if f in ("search", "grover_qft"):
        st["s"] = qc.State(case["n"], case["dt"])
        st["marked"] = W.marked_indices(_rng(seed), case["n"], case["marked"])
    elif f == "shor":
        st["n1"], st["n2"], st["x"] = _shor(case, seed)
        st["s"] = qc.State(st["n1"] + st["n2"], case["dt"])
    elif f in ("qft", "circuit", "fused", "hamiltonian", "measure"):
        st["s"] = qc.State(case["n"], case["dt"], tensor=_state(case["n"], seed, case["dt"]))
        if f == "circuit":
            st["layers"] = _circuit(case, seed)
        elif f == "fused":
            k, pad = (5, True) if case["dt"] == C64 else (3, False)
            st["plan"] = qc.FusedPlan(case["n"], _fused_ops(case, seed), kmax=min(k, case["n"]), pad=pad)
        elif f == "hamiltonian":
            st["terms"] = _chain(case, seed)
        elif f == "measure":
            st["strings"] = _strings(case, seed)
    elif f == "adjoint":
        gates, terms = _ansatz(case)
        st["circuit"] = qc.Circuit(case["n"], gates, terms, dt=case["dt"])
        st["theta"] = _theta(case, seed).requires_grad_(True)
    elif f == "traj":
        b = W.trajectory_batch(case["inst"], case["n_lo"], case["n_hi"], seed & 0x7FFFFFFF, case["p"], case["p"])
        # the built-in launch shape: which one a timed search would pick
        # differs from run to run
        st["plan"] = qc.TrajectoryPlan(b.nq, b.marked, b.iters, b.seed, b.p_gate, b.p_readout, autotune=False)
    elif f == "rho":
        st["psi"], st["P"] = _ensemble(case, seed)
        st["rho"] = torch.empty((1 << case["n"], 1 << case["n"]), dtype=st["psi"].dtype, device="cuda")
    return st


# ------------------------------------------------------------------ passes --

def run(st):
    case = st["case"]
    f = case["family"]
    if f == "search":
        s = st["s"]
        s.grover_run(st["marked"], case["iters"])
        if case["dt"] == C64:
            return [s.tensor]
        p, shots = s.probs_sample(st["seed"], case["shots"])
        return [s.tensor, p, shots]
    if f == "shor":
        s = st["s"]
        qc.qc_shor_prepare(s.h, st["n2"], st["x"], case["M"])
        prob = qc.qc_project(s.h, 0, st["n2"], st["x"])
        qc.qc_qft_range(s.h, st["n2"], st["n1"])
        if case["dt"] == C64:
            return [prob, s.tensor]
        p, shots = s.probs_sample(st["seed"], case["shots"])
        return [prob, s.tensor, p, shots]
    if f == "grover_qft":
        s = st["s"]
        s.uniform()
        for _ in range(case["iters"]):
            s.grover_step(st["marked"])
        s.qft()
        if case["dt"] == C64:
            return [s.tensor]
        p, shots = s.probs_sample(st["seed"], case["shots"])
        return [s.tensor, p, shots]
    if f == "qft":
        st["s"].qft()
        return [st["s"].tensor]
    if f == "circuit":
        s = st["s"]
        for U, pairs in st["layers"]:
            for q in range(case["n"]):
                s.apply_1q(q, U[q])
            for c, t in pairs:
                s.cnot(c, t)
        return [s.tensor]
    if f == "fused":
        st["plan"].run(st["s"].h)
        return [st["s"].tensor]
    if f == "hamiltonian":
        for _ in range(case["steps"]):
            qc.qc_hamiltonian_step(st["s"].h, 1e-2, st["terms"])
        return [st["s"].tensor]
    if f == "measure":
        s = st["s"]
        norm = s.renormalize()
        e = [s.expect_pauli(x, z).real for x, z in st["strings"]]
        p, shots = s.probs_sample(st["seed"], case["shots"])
        return [norm, np.array(e), s.tensor, p, shots]
    if f == "adjoint":
        theta = st["theta"]
        theta.grad = None
        E = qc.energy(theta, st["circuit"])
        E.sum().backward()
        return [E.detach(), theta.grad]
    if f == "traj":
        o = st["plan"].run()
        return [o["p_success"], o["p_readout"], o["outcome"], o["n_errors"]]
    if f == "rho":
        psi, rho = st["psi"], st["rho"]
        stream = torch.cuda.current_stream().cuda_stream
        qc.qc_density_matrix(psi.data_ptr(), case["n"], case["dt"], case["batch"], st["P"], rho.data_ptr(), stream)
        ev, stats = qc.qc_mixed_spectrum(psi.data_ptr(), case["n"], case["dt"], case["batch"], st["P"], stream)
        return [rho, ev, np.array(stats)]
    raise ValueError(f)


# -------------------------------------------------------------------- work --

def work(case):
    """What one pass cannot do without: a call on a state reads and writes the
    amplitudes its operator touches once; arithmetic as the operator needs."""
    f = case["family"]
    ab = 8 if case.get("dt") == C64 else 16
    if f == "shor":
        n1, n2, _ = _shor(case, 0)
        N = 1 << (n1 + n2)
        # write the state; write it projected (and read the outcome); QFT; probabilities
        b = ab * (N + N + 2 * N) + (0 if case["dt"] == C64 else ab * N + 8 * N)
        return dict(bytes=b, flops=N * (5 * n1 + 8))
    if f == "traj":
        nq = [n for n in range(case["n_lo"], case["n_hi"] + 1)]
        per = case["inst"] / len(nq)
        # an error-free stretch needs no pass over the state; one with errors reads and writes it
        it = [(n, W.grover_iterations(n)) for n in nq]
        b = sum(per * 16 * 2.0 ** n * i * (1 - (1 - case["p"]) ** (2 * n + 1)) for n, i in it)
        return dict(bytes=b, flops=b)
    n = case["n"]
    N = 1 << n
    S = ab * N
    if f == "search":
        return dict(bytes=S + (0 if case["dt"] == C64 else 8 * N), flops=4.0 * N * case["iters"] + 4 * N)
    if f == "grover_qft":
        b = S + 2 * S * case["iters"] + 2 * S + (0 if case["dt"] == C64 else S + 8 * N)
        return dict(bytes=b, flops=N * (4.0 * case["iters"] + 5 * n))
    if f == "qft":
        return dict(bytes=2 * S, flops=5.0 * n * N)
    if f == "circuit":
        cn = sum(len(range(l % 2, n - 1, 2)) for l in range(case["layers"]))
        return dict(bytes=2 * S * n * case["layers"] + S * cn, flops=14.0 * N * n * case["layers"])
    if f == "fused":
        # a pass over the state for every five (three) qubits of a layer
        k = 5 if case["dt"] == C64 else 3
        blocks = case["layers"] * math.ceil(n / k)
        return dict(bytes=2 * S * blocks, flops=14.0 * N * n * case["layers"])
    if f == "hamiltonian":
        # the state is read and written once a step; a chain's terms cost about 6 complex multiply-adds an amplitude and site
        return dict(bytes=2 * S * case["steps"], flops=48.0 * N * n * case["steps"])
    if f == "measure":
        # scale, every string and the read-out read the state once; scale and probabilities write
        return dict(bytes=S + 2 * S + S * case["terms"] + S + 8 * N, flops=N * (8.0 + 8.0 * case["terms"]))
    if f == "adjoint":
        # a layer's ring mixes all qubits: the forward sweep reads and writes psi
        # once a layer, the backward sweep psi and lambda
        B, L = case["batch"], case["layers"]
        return dict(bytes=B * S * L * (2 + 4), flops=B * N * L * n * (14.0 + 2 * 14.0 + 2 * 8.0))
    if f == "rho":
        B = case["batch"]
        return dict(bytes=B * S + ab * 4.0 ** n + B * S, flops=4.0 ** n * B * 4 + 8.0 * B * B * N / 2)
    raise ValueError(f)


# ------------------------------------------------------- values in 64 bits --

def _apply(v, n, qubits, m):
    """A matrix on `qubits` (local bit b on qubits[b]) of v (..., 2^n)."""
    k = len(qubits)
    lead = v.dim() - 1
    t = v.reshape(v.shape[:-1] + (2,) * n)
    axes = [lead + n - 1 - q for q in reversed(qubits)]  # most significant local bit first
    m = torch.as_tensor(np.asarray(m, dtype=np.complex128), device=v.device).reshape((2,) * (2 * k))
    r = torch.tensordot(m, t, dims=(list(range(k, 2 * k)), axes))
    return torch.movedim(r, list(range(k)), axes).reshape(v.shape)


def _pair(v, n, q, m):
    """A 2x2 matrix, or one for each row of v (B, 2^n), on qubit q."""
    B = v.shape[0]
    t = v.view(B, 1 << (n - 1 - q), 2, 1 << q)
    c = [[m[..., i, j].reshape(-1, 1, 1) for j in range(2)] for i in range(2)]
    a, b = t[:, :, 0], t[:, :, 1]
    return torch.stack([c[0][0] * a + c[0][1] * b, c[1][0] * a + c[1][1] * b], dim=2).view(B, 1 << n)


def _cnot_index(n, pairs, device):
    """The gather index of CNOTs applied in order: new[j] = old[index[j]]."""
    j = torch.arange(1 << n, device=device)
    for c, t in reversed(pairs):
        j = j ^ (((j >> c) & 1) << t)
    return j


def _idft(v, lo, width, n):
    """2^{-w/2} sum e^{+2 pi i jk / 2^w} on the register [lo, lo + width)."""
    t = v.view(1 << (n - lo - width), 1 << width, 1 << lo)
    return torch.fft.ifft(t, dim=1, norm="ortho").reshape(-1)


def _rot(kind, theta):
    c, s = torch.cos(theta / 2).to(torch.complex128), torch.sin(theta / 2).to(torch.complex128)
    z = torch.zeros_like(c)
    if kind == "y":
        rows = [torch.stack([c, -s], -1), torch.stack([s, c], -1)]
    else:
        rows = [torch.stack([c - 1j * s, z], -1), torch.stack([z, c + 1j * s], -1)]
    return torch.stack(rows, -2)


def _exact_adjoint(case, theta):
    n, L, B = case["n"], case["layers"], theta.shape[0]
    th = theta.detach().to(torch.float64).view(B, L, n, 2)
    ring = _cnot_index(n, [(q, (q + 1) % n) for q in range(n)], theta.device)
    back = torch.empty_like(ring)
    back[ring] = torch.arange(1 << n, device=ring.device)
    v = torch.zeros((B, 1 << n), dtype=torch.complex128, device=theta.device)
    v[:, 0] = 1
    for l in range(L):
        for q in range(n):
            v = _pair(v, n, q, _rot("z", th[:, l, q, 1]) @ _rot("y", th[:, l, q, 0]))
        v = v[:, ring]
    j = torch.arange(1 << n, device=theta.device)
    lam = torch.zeros_like(v)
    for x, z, c in W.ansatz_hamiltonian(n):  # no Y factors
        par = torch.zeros_like(j)
        for q in range(n):
            if (z >> q) & 1:
                par ^= (j >> q) & 1
        lam += c * (1 - 2 * par).to(torch.float64) * v[:, j ^ x]
    E = (v.conj() * lam).sum(dim=1).real
    grad = torch.empty((B, L, n, 2), dtype=torch.float64, device=theta.device)
    for l in reversed(range(L)):
        v, lam = v[:, back], lam[:, back]
        for q in reversed(range(n)):
            for k, kind in ((1, "z"), (0, "y")):
                p, w = (a.view(B, -1, 2, 1 << q) for a in (v, lam))
                if kind == "z":
                    d = (w[:, :, 0].conj() * p[:, :, 0] - w[:, :, 1].conj() * p[:, :, 1]).sum(dim=(1, 2))
                else:
                    d = (-1j * w[:, :, 0].conj() * p[:, :, 1] + 1j * w[:, :, 1].conj() * p[:, :, 0]).sum(dim=(1, 2))
                grad[:, l, q, k] = d.imag
                m = _rot(kind, -th[:, l, q, k])
                v, lam = _pair(v, n, q, m), _pair(lam, n, q, m)
    return [E, grad.view(B, -1)]


def _exact_search(case, marked, iters):
    """The closed form of `iters` Grover operators on the uniform state."""
    N, M = 1 << case["n"], len(marked)
    t = math.asin(math.sqrt(M / N))
    a, b = math.sin((2 * iters + 1) * t) / math.sqrt(M), math.cos((2 * iters + 1) * t) / math.sqrt(N - M)
    v = torch.full((N,), b, dtype=torch.complex128, device="cuda")
    v[torch.as_tensor(marked.astype(np.int64), device="cuda")] = a
    return v


def _born(v):
    r = torch.view_as_real(v)
    return r[..., 0].square() + r[..., 1].square()


def exact(case, seed):
    f = case["family"]
    wide = case.get("dt") == C128
    if f == "traj":
        return None  # noise strikes gate by gate: a plain replay takes minutes
    if f in ("search", "grover_qft"):
        v = _exact_search(case, W.marked_indices(_rng(seed), case["n"], case["marked"]), case["iters"])
        if f == "grover_qft":
            v = torch.fft.ifft(v, norm="ortho")
        return [v, _born(v), None] if wide else [v]
    if f == "shor":
        n1, n2, x = _shor(case, seed)
        M, y, hits = case["M"], 1, []
        for j in range(1 << n1):
            if y == x:
                hits.append((j << n2) | y)
            y = y * x % M
        v = torch.zeros(1 << (n1 + n2), dtype=torch.complex128, device="cuda")
        v[torch.tensor(hits, device="cuda")] = 1 / math.sqrt(len(hits))
        v = _idft(v, n2, n1, n1 + n2)
        prob = len(hits) / (1 << n1)
        return [prob, v, _born(v), None] if wide else [prob, v]
    if f == "adjoint":
        return _exact_adjoint(case, _theta(case, seed))
    if f == "rho":
        psi, P = _ensemble(case, seed)
        v = psi.to(torch.complex128) * torch.as_tensor(P, device="cuda").sqrt()[:, None]
        rho = v.T @ v.conj()
        ev = torch.linalg.eigvalsh(v.conj() @ v.T).flip(0).cpu().numpy()
        pos = ev[ev > 1e-14]
        return [rho, ev, np.array([ev.sum(), (ev * ev).sum(), -(pos * np.log(pos)).sum()])]
    n = case["n"]
    v = _state(n, seed, case["dt"]).to(torch.complex128)
    if f == "qft":
        return [torch.fft.ifft(v, norm="ortho")]
    if f in ("circuit", "fused"):
        for U, pairs in _circuit(case, seed):
            for q in range(n):
                m = U[q].reshape(2, 2, 2)
                m = torch.as_tensor(m[..., 0] + 1j * m[..., 1], device="cuda")
                v = _pair(v.view(1, -1), n, q, m).view(-1)
            v = v[_cnot_index(n, pairs, "cuda")]
        return [v]
    if f == "hamiltonian":
        terms = _chain(case, seed)
        for _ in range(case["steps"]):
            d = torch.zeros_like(v)
            for qs, m in terms:
                d += _apply(v, n, qs, m)
            v = v - 1e-2j * d
        return [v]
    if f == "measure":
        norm = _born(v).sum()
        v = v / norm.sqrt()
        j = torch.arange(1 << n, device="cuda")
        e = []
        for x, z in _strings(case, seed):
            par = torch.zeros_like(j)
            for q in range(n):
                if (z >> q) & 1:
                    par ^= (j >> q) & 1
            # P|j> = i^{|x&z|} (-1)^{|j&z|} |j^x>
            w = (1j ** bin(x & z).count("1")) * (1 - 2 * par).to(torch.float64) * v
            e.append(float((v[j ^ x].conj() * w).sum().real))
        return [float(norm), np.array(e), v, _born(v), None]
    raise ValueError(f)
