"""The work that is timed when this library's speed is judged: circuits run through the public entry points.

A case is a dict of plain values; ``kind`` says which entry points it goes through:

  gates    single ``State.apply_gate`` calls on a state a program holds (interactive use)
  oneshot  ``State.run`` from |0...0> with planning in the call, then ``State.expect_z`` (a variational loop)
  plan     a kept ``Plan`` executed from a basis state (repeated runs of one circuit)
  batch    a kept ``Batch`` of TFIM chains executed, its <Z> statistics read back
  readout  <Z> statistics with samples, a marginal, Pauli strings and the norm of a state in hand

Circuits come from ``workloads`` (the families the paper benchmarks); ``exact`` applies the same gate lists with
plain torch in 64 bits.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import workloads as W
from paper_2511_14664_gb300 import qsim

PRECISION = {"simt": qsim.PREC_SIMT, "tf32x3": qsim.PREC_TF32X3, "fp16x3": qsim.PREC_FP16X3}


def listed():
    return [
        # one layer of gates called one by one on a small state: what a notebook or a debugger does
        dict(name="gates_n10", kind="gates", n=10, dtype="c64"),
        # one step of a variational loop: a new 12-qubit circuit planned, run and read out in single calls
        dict(name="oneshot_tfim_n12", kind="oneshot", family="tfim", n=12, depth=6, dtype="c64", mode="fused",
             max_fused=5, precision="simt"),
        # the 14-qubit double-precision brickwork of the benchmark (410 gates), full vector
        dict(name="brick_n14_c128", kind="plan", family="brickwork", n=14, depth=20, dtype="c128", mode="fused",
             max_fused=5, precision="simt"),
        # a medium single-precision brickwork: the whole state stays in L2
        dict(name="brick_n21_fp16x3", kind="plan", family="brickwork", n=21, depth=40, dtype="c64", mode="fused",
             max_fused=7, precision="fp16x3"),
        # the headline of the benchmark: 30 qubits, depth 40, 1780 gates
        dict(name="brick_n30_fp16x3", kind="plan", family="brickwork", n=30, depth=40, dtype="c64", mode="fused",
             max_fused=7, precision="fp16x3"),
        # the QFT of the benchmark from a basis state (dense blocks with long runs of controlled phases)
        dict(name="qft_n28_fp16x3", kind="plan", family="qft", n=28, depth=0, dtype="c64", mode="fused",
             max_fused=6, precision="fp16x3"),
        # the paper's random circuit (30 n gates on random qubits), odd width, fused tensor-core blocks
        dict(name="rcs_n27_tf32x3", kind="plan", family="rcs", n=27, depth=30, dtype="c64", mode="fused",
             max_fused=6, precision="tf32x3"),
        # the same circuit family gate by gate (the default mode of State.run and Plan)
        dict(name="rcs_n25_plain", kind="plan", family="rcs", n=25, depth=30, dtype="c64", mode="plain",
             max_fused=5, precision="simt"),
        # default fused options (5-qubit blocks, single-precision arithmetic) on random Haar U(4) pairs
        dict(name="pairs_n26_simt", kind="plan", family="pairs", n=26, depth=16, dtype="c64", mode="fused",
             max_fused=5, precision="simt"),
        # a double-precision circuit larger than the caches, default fused options
        dict(name="brick_n23_c128", kind="plan", family="brickwork", n=23, depth=10, dtype="c128", mode="fused",
             max_fused=5, precision="simt"),
        # many independent TFIM chains of mixed width in one call (iterative algorithms, parameter scans)
        dict(name="batch_64_n10_24", kind="batch", count=64, nmin=10, nmax=24, smin=8, smax=32, precision="fp16x3"),
        # everything a program reads from a large state: <Z>, <ZZ>, 1000 samples, a marginal, Pauli strings, norm
        dict(name="readout_n28", kind="readout", n=28, dtype="c64", shots=1000, marginal=12),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["gates", "oneshot", "plan", "plan", "plan", "plan", "plan", "batch", "readout", "readout"])
    if kind == "gates":
        return dict(kind=kind, n=rng.randint(4, 22), dtype=rng.choice(["c64", "c128"]))
    if kind == "oneshot":
        return dict(kind=kind, family=rng.choice(["tfim", "brickwork", "rcs"]), n=rng.randint(5, 18),
                    depth=rng.randint(2, 10), dtype=rng.choice(["c64", "c128"]), mode=rng.choice(["plain", "fused"]),
                    max_fused=rng.randint(3, 5), precision="simt")
    if kind == "batch":
        nmin = rng.randint(6, 14)
        return dict(kind=kind, count=rng.randint(8, 64), nmin=nmin, nmax=rng.randint(nmin + 2, 24), smin=4,
                    smax=rng.randint(8, 32), precision=rng.choice(["simt", "tf32x3", "fp16x3"]))
    if kind == "readout":
        dtype = rng.choice(["c64", "c64", "c128"])
        n = rng.randint(8, 29 if dtype == "c64" else 27)
        return dict(kind=kind, n=n, dtype=dtype, shots=rng.choice([100, 1000, 10000]),
                    marginal=rng.randint(1, min(n, 14)))
    family = rng.choice(["brickwork", "rcs", "pairs", "qft", "tfim"])
    how = rng.choice(["tc", "tc", "simt", "plain", "c128"])
    if how == "tc":
        precision = rng.choice(["fp16x3", "tf32x3"])
        n, depth, dtype, mode = rng.randint(14, 28), rng.randint(8, 40), "c64", "fused"
        max_fused = rng.randint(5, 7 if precision == "fp16x3" else 6)
    elif how == "simt":
        precision, n, depth, dtype, mode = "simt", rng.randint(10, 26), rng.randint(4, 20), "c64", "fused"
        max_fused = rng.randint(3, 6)
    elif how == "plain":
        precision, dtype, mode, max_fused = "simt", rng.choice(["c64", "c64", "c128"]), "plain", 5
        n, depth = rng.randint(10, 26 if dtype == "c64" else 23), rng.randint(4, 20)
    else:
        precision, n, depth, dtype, mode = "simt", rng.randint(10, 23), rng.randint(4, 12), "c128", "fused"
        max_fused = rng.randint(3, 6)
    return dict(kind="plan", family=family, n=n, depth=0 if family == "qft" else depth, dtype=dtype, mode=mode,
                max_fused=max_fused, precision=precision)


# -- inputs -----------------------------------------------------------------------------------------------------
def _circuit(case, seed):
    n, d = case["n"], case["depth"]
    if case["family"] == "brickwork":
        return W.brickwork(n, d, seed)
    if case["family"] == "rcs":
        return W.rcs(n, seed, gates_per_qubit=d)
    if case["family"] == "pairs":
        return W.random_pairs(n, d, seed)
    if case["family"] == "qft":
        return W.qft(n)
    rng = np.random.default_rng(seed)
    return W.tfim_chain(n, d, float(rng.uniform(0, math.pi)), float(rng.uniform(0, math.pi)))


def _layer(n, seed):
    """A rotation on every qubit and a chain of controlled-NOTs, as (targets, controls, matrix)."""
    rng = np.random.default_rng(seed)
    out = [((q,), (), W.haar_unitary(2, rng)) for q in range(n)]
    return out + [((q + 1,), (q,), W.X()) for q in range(n - 1)]


def _chains(case, seed):
    """The TFIM chains of a batch: their widths and depths belong to the case, their angles to the seed."""
    shape, rng = np.random.default_rng(case["count"]), np.random.default_rng(seed)
    return [W.tfim_chain(int(shape.integers(case["nmin"], case["nmax"] + 1)),
                         int(shape.integers(case["smin"], case["smax"] + 1)),
                         float(rng.uniform(0, math.pi)), float(rng.uniform(0, math.pi)))
            for _ in range(case["count"])]


def _basis(case, seed):
    """The basis state a plan starts from: |0...0>, or a seeded one for the QFT (whose circuit is fixed)."""
    return W.basis_index(case["n"], seed) if case["family"] == "qft" else 0


def _random_state(case, seed):
    """A normalised state with Gaussian amplitudes (as a deep random circuit gives) under a product envelope, so
    that every qubit has a magnetisation of its own."""
    n = case["n"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    real = torch.float32 if case["dtype"] == "c64" else torch.float64
    psi = torch.randn(1 << n, 2, dtype=real, device="cuda", generator=g)
    rng = np.random.default_rng(seed)
    for q in range(n):
        th = float(rng.uniform(0.15 * math.pi, 0.35 * math.pi))
        v = psi.view(1 << (n - 1 - q), 2, 2 << q)
        v[:, 0] *= math.sqrt(2) * math.cos(th)
        v[:, 1] *= math.sqrt(2) * math.sin(th)
    psi /= float(psi.view(-1).double().square().sum().sqrt())
    return torch.view_as_complex(psi)


def _readout_inputs(case, seed):
    """The marginal's qubits and two Pauli strings: one of Z alone, one mixed."""
    rng = np.random.default_rng(seed + 1)
    n = case["n"]
    qubits = [int(q) for q in rng.permutation(n)[: case["marginal"]]]
    return qubits, ["".join(rng.choice(list("IZ"), n)), "".join(rng.choice(list("IXYZ"), n))]


def _state(case, tensor=None):
    return qsim.State(case["n"], qsim.C64 if case["dtype"] == "c64" else qsim.C128, tensor=tensor)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gates":
        st = _state(case)
        st.set_basis(0)
        return dict(kind=kind, st=st, gates=_layer(case["n"], seed))
    if kind == "readout":
        qubits, strings = _readout_inputs(case, seed)
        return dict(kind=kind, st=_state(case, _random_state(case, seed)), seed=seed, shots=case["shots"],
                    qubits=qubits, strings=strings)
    if kind == "batch":
        return dict(kind=kind, batch=qsim.Batch(_chains(case, seed), precision=PRECISION[case["precision"]]))
    opts = dict(mode=qsim.RUN_FUSED if case["mode"] == "fused" else qsim.RUN_PLAIN, max_fused=case["max_fused"],
                precision=PRECISION[case["precision"]])
    st = _state(case)
    circuit = _circuit(case, seed)
    if kind == "oneshot":
        return dict(kind=kind, st=st, circuit=circuit, opts=opts, dtype=case["dtype"])
    return dict(kind=kind, st=st, plan=qsim.Plan(circuit, dtype=st.dtype, **opts), x=_basis(case, seed))


# -- one pass ----------------------------------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "gates":
        st = state["st"]
        for targets, controls, u in state["gates"]:
            st.apply_gate(targets, controls, u)
        return st.tensor
    if kind == "oneshot":
        st = state["st"]
        st.set_basis(0)
        st.run(state["circuit"], **state["opts"])
        zi, zz = st.expect_z()
        real = np.float32 if state["dtype"] == "c64" else np.float64  # as exact as the amplitudes they come from
        return [st.tensor, zi.astype(real), zz.astype(real)]
    if kind == "plan":
        state["plan"].execute_from_basis(state["st"], state["x"])
        return state["st"].tensor
    if kind == "batch":
        b = state["batch"]
        b.execute()
        res = b.results()  # from complex64 states: single precision is what the values carry
        return [np.concatenate([z for z, _ in res]).astype(np.float32),
                np.concatenate([zz for _, zz in res]).astype(np.float32)]
    st = state["st"]
    zi, zz, samples = st.expect_z_and_sample(state["seed"], state["shots"])
    return [zi, zz, samples.view(np.int64), st.probs(state["qubits"]),
            np.array([st.expect_pauli(p) for p in state["strings"]]), st.norm()]


# -- what a pass cannot do without --------------------------------------------------------------------------------
def _gate_flops(n, targets, controls, u):
    """Complex multiply-adds of one gate, gate by gate: 8 flops each, on the amplitudes it touches."""
    u = np.asarray(u)
    per_group = 8.0 * np.count_nonzero(u) if np.count_nonzero(u - np.diag(np.diag(u))) \
        else 6.0 * np.count_nonzero(np.diag(u) != 1)
    return float(per_group) * 2.0 ** (n - len(targets) - len(controls))


def _circuit_flops(c):
    memo, total = {}, 0.0  # circuits share matrix objects between gates
    for g in c.gates:
        key = (id(g.matrix), len(g.controls))
        if key not in memo:
            memo[key] = _gate_flops(c.n, g.targets, g.controls, g.matrix)
        total += memo[key]
    return total


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # every chain's gates; the states need never leave the chip, so the bytes are the <Z> values alone
        circuits = _chains(case, 1)
        return dict(bytes=sum(8.0 * (2 * c.n - 1) for c in circuits), flops=sum(_circuit_flops(c) for c in circuits))
    state_bytes = 2.0 ** case["n"] * (8 if case["dtype"] == "c64" else 16)
    if kind == "gates":  # the state read and written once for the layer
        return dict(bytes=2 * state_bytes,
                    flops=sum(_gate_flops(case["n"], t, c, u) for t, c, u in _layer(case["n"], 1)))
    if kind == "readout":  # the state read once; |a|^2 and a signed sum for every value that is wanted
        return dict(bytes=state_bytes + 8 * 2.0 ** case["marginal"] + 8 * case["shots"],
                    flops=2.0 ** case["n"] * (4 + 2 * case["n"] + 16))
    # from a basis state: the state is written once
    return dict(bytes=state_bytes, flops=_circuit_flops(_circuit(case, 1)))


# -- the same results in 64 bits ----------------------------------------------------------------------------------
def _apply(psi, n, targets, controls, u):
    """Apply u to psi (2^n complex128 amplitudes) in place."""
    qs = sorted(tuple(targets) + tuple(controls), reverse=True)
    shape, top = [], n
    for q in qs:
        shape += [1 << (top - 1 - q), 2]
        top = q
    v = psi.view(shape + [1 << top])
    where = {q: 2 * i + 1 for i, q in enumerate(qs)}
    sub = []
    for m in range(1 << len(targets)):
        index = [slice(None)] * v.dim()
        for q in controls:
            index[where[q]] = 1
        for j, q in enumerate(targets):
            index[where[q]] = (m >> j) & 1
        sub.append(v[tuple(index)])
    u = np.asarray(u)
    if np.count_nonzero(u - np.diag(np.diag(u))) == 0:
        for m, s in enumerate(sub):
            if u[m, m] != 1:
                s.mul_(complex(u[m, m]))
        return
    old = [s.clone() for s in sub]
    for r, s in enumerate(sub):
        s.zero_()
        for c, o in enumerate(old):
            if u[r, c] != 0:
                s.add_(o, alpha=complex(u[r, c]))


def _evolve(n, gates, x=0):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[x] = 1
    for targets, controls, u in gates:
        _apply(psi, n, targets, controls, u)
    return psi


def _z(psi, n):
    """<Z_i> and <Z_i Z_i+1> of a state, 64 bits."""
    p = psi.real.square() + psi.imag.square()
    zi, zz = [], []
    for q in range(n):
        v = p.view(1 << (n - 1 - q), 2, 1 << q)
        zi.append(float(v[:, 0].sum() - v[:, 1].sum()))
    for q in range(n - 1):
        v = p.view(1 << (n - 2 - q), 2, 2, 1 << q)
        zz.append(float(v[:, 0, 0].sum() - v[:, 0, 1].sum() - v[:, 1, 0].sum() + v[:, 1, 1].sum()))
    return np.array(zi), np.array(zz)


def _pauli(psi, n, string):
    """<P> of a Pauli string."""
    out = psi.clone()
    mats = dict(X=W.X(), Y=W.Y(), Z=W.Z())
    for q, p in enumerate(string):
        if p != "I":
            _apply(out, n, (q,), (), mats[p])
    return complex(torch.vdot(psi, out))


def _marginal(psi, n, qubits):
    p = (psi.real.square() + psi.imag.square()).cpu().numpy()
    m = np.zeros(1, dtype=np.int64)
    for q in range(n):  # bin of every index, bit by bit
        j = qubits.index(q) if q in qubits else None
        m = np.concatenate([m, m + (0 if j is None else 1 << j)])
    return np.bincount(m, weights=p, minlength=1 << len(qubits))


def exact(case, seed):
    kind, n = case["kind"], case.get("n")
    if kind == "gates":
        return _evolve(n, _layer(n, seed))
    if kind == "batch":
        res = [_z(_evolve(c.n, [(g.targets, g.controls, g.matrix) for g in c.gates]), c.n)
               for c in _chains(case, seed)]
        return [np.concatenate([z for z, _ in res]), np.concatenate([zz for _, zz in res])]
    if kind == "readout":
        psi = _random_state(case, seed).to(torch.complex128)
        qubits, strings = _readout_inputs(case, seed)
        zi, zz = _z(psi, n)
        return [zi, zz, None, _marginal(psi, n, qubits), np.array([_pauli(psi, n, s) for s in strings]),
                float(psi.real.square().sum() + psi.imag.square().sum())]
    if kind == "plan" and n > 28:
        return None  # 64-bit gate by gate at 30 qubits takes minutes
    if kind == "plan" and case["family"] == "qft":
        y = torch.arange(1 << n, dtype=torch.int64, device="cuda")
        turn = ((y * _basis(case, seed)) & ((1 << n) - 1)).double() * (2 * math.pi / (1 << n))
        return torch.polar(torch.full_like(turn, 2.0 ** (-n / 2)), turn)
    circuit = _circuit(case, seed)
    psi = _evolve(n, [(g.targets, g.controls, g.matrix) for g in circuit.gates], 0)
    if kind == "oneshot":
        return [psi, *_z(psi, n)]
    return psi
