"""Per-gate plans whose gates run many to a pass (tiles in shared memory) against the FP64 oracle.

Tolerance as for the other per-gate paths: complex64 max |amplitude error| <= 1e-5 and normalised infidelity <= 1e-9,
complex128 <= 1e-12 and <= 1e-12.
"""
import numpy as np
import pytest

import oracle
import workloads as W
from helpers import random_state

pytestmark = pytest.mark.gpu

C64, C128 = 0, 1
TOL = {C64: (1e-5, 1e-9), C128: (1e-12, 1e-12)}


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


def mixed(n, gates, seed):
    """Every form a group takes and some it does not: dense gates on 1..3 targets, real and imaginary ones, swaps,
    diagonals on 1..3 qubits, controls on any qubit."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for _ in range(gates):
        kind = int(rng.integers(0, 8))
        q = [int(x) for x in rng.permutation(n)[:5]]
        th = float(rng.uniform(0, 6))
        if kind == 0:
            c.append(W.Gate((q[0],), (), W.haar_unitary(2, rng), "u"))
        elif kind == 1:
            c.append(W.Gate((q[0],), tuple(q[1:1 + int(rng.integers(0, 3))]), (W.RY, W.RX)[int(rng.integers(0, 2))](th), "r"))
        elif kind == 2:
            c.append(W.Gate((q[0], q[1]), tuple(q[2:2 + int(rng.integers(0, 2))]), W.haar_unitary(4, rng), "u4"))
        elif kind == 3:
            c.append(W.Gate((q[0], q[1]), (), W.SWAP(), "swap"))
        elif kind == 4:
            c.append(W.Gate((q[0],), (q[1],), W.CP(th), "cp"))
        elif kind == 5:
            c.append(W.Gate((q[0], q[1]), (), W.RZZ(th), "rzz"))
        elif kind == 6:
            c.append(W.random_gate(n, rng, kmax=3, cmax=2, diag_prob=0.5))
        else:
            c.append(W.Gate((q[0],), (q[1],), W.X(), "cx"))
    return c


def check(g, ref, n, dtype):
    at, it = TOL[dtype]
    g = np.ascontiguousarray(g.astype(np.complex128))
    assert float(np.max(np.abs(g - ref))) <= at
    assert oracle.infidelity(g, ref, n) <= it


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n,gates", [(17, 2), (17, 150), (18, 400), (20, 120), (21, 60)])
def test_mixed_circuits(qsim, dtype, n, gates):
    """One to several tiles per CTA, one gate to programs cut at their size limit; twice from a given state, and from
    a basis state."""
    c = mixed(n, gates, seed=n + gates)
    p = qsim.Plan(c, dtype, mode=0)
    assert p.info["passes"] == len(c)
    psi0 = random_state(n, 5)
    psi0 = psi0.astype(np.complex64) if dtype == C64 else psi0
    st = qsim.State(n, dtype)
    st.set_state(psi0)
    p.execute(st)
    ref = oracle.run(c, psi=psi0.astype(np.complex128))
    check(st.get_state(), ref, n, dtype)
    p.execute_from_basis(st, 3)
    check(st.get_state(), oracle.run(c, basis_state=3), n, dtype)


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("make", [lambda: W.qft(17), lambda: W.rcs(17, 3), lambda: W.brickwork(18, 12, 4),
                                  lambda: W.tfim_chain(17, 6, 0.3, 0.8), lambda: W.ghz(19)])
def test_circuit_families(qsim, dtype, make):
    c = make()
    st = qsim.State(c.n, dtype)
    st.set_basis(1)
    st.run(c, mode=0)
    check(st.get_state(), oracle.run(c, basis_state=1), c.n, dtype)


@pytest.mark.parametrize("dtype", [C64, C128])
def test_equals_the_passes_one_by_one(qsim, dtype):
    """Executed pass by pass the same plan runs one kernel a gate; the results agree to the reordering of commuting
    gates, and a pass range still means those gates."""
    n, c = 18, mixed(18, 80, seed=9)
    p = qsim.Plan(c, dtype, mode=0)
    a, b = qsim.State(n, dtype), qsim.State(n, dtype)
    psi0 = random_state(n, 6).astype(np.complex64 if dtype == C64 else np.complex128)
    a.set_state(psi0)
    b.set_state(psi0)
    p.execute(a)
    p.execute_range(b, 0, 30)
    p.execute_range(b, 30, len(c) - 30)
    check(a.get_state(), b.get_state().astype(np.complex128), n, dtype)
