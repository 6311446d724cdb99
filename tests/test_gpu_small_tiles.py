"""Small states' plans that run many gates between two grid barriers against the FP64 oracle.

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
    """Dense gates on 1 and 2 targets (general, real, RX, swap), diagonals, controls on any qubit."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for _ in range(gates):
        q = [int(x) for x in rng.permutation(n)]
        th = float(rng.uniform(0, 6))
        kind = int(rng.integers(0, 7))
        if n == 1 or kind == 0:
            c.append(W.Gate((q[0],), (), (W.haar_unitary(2, rng), W.RX(th), W.RZ(th))[int(rng.integers(0, 3))], "u"))
        elif kind == 1:
            c.append(W.Gate((q[0],), tuple(q[1:1 + int(rng.integers(0, 3))]), (W.RY, W.RX)[int(rng.integers(0, 2))](th), "r"))
        elif kind == 2:
            c.append(W.Gate((q[0], q[1]), tuple(q[2:2 + int(rng.integers(0, 2))]), W.haar_unitary(4, rng), "u4"))
        elif kind == 3:
            c.append(W.Gate((q[0], q[1]), (), W.SWAP(), "swap"))
        elif kind == 4:
            c.append(W.Gate((q[0],), (q[1],), W.CP(th) if n % 2 else W.CP(np.pi), "cp"))
        elif kind == 5:
            c.append(W.Gate((q[0], q[1]), (), W.RZZ(th), "rzz"))
        else:
            c.append(W.Gate((q[0],), (q[1],), W.X(), "cx"))
    return c


def check(g, ref, n, dtype):
    at, it = TOL[dtype]
    g = np.ascontiguousarray(g.astype(np.complex128))
    assert float(np.max(np.abs(g - ref))) <= at
    assert oracle.infidelity(g, ref, n) <= it


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n", [1, 2, 5, 6, 7, 8, 9, 10, 14, 15, 16])
def test_modes_and_entries(qsim, dtype, n):
    c = mixed(n, 60, seed=400 + 2 * n + dtype)
    psi0 = random_state(n, 4)
    psi0 = psi0.astype(np.complex64) if dtype == C64 else psi0
    ref = oracle.run(c, psi=psi0.astype(np.complex128))
    ref2 = oracle.run(c, psi=ref.copy())
    x = (1 << n) - 2 if n > 1 else 1
    base = oracle.run(c, basis_state=x)
    for mode in (0, 1):
        st = qsim.State(n, dtype)
        plan = qsim.Plan(c, dtype, mode=mode, max_fused=4)
        st.set_state(psi0)
        plan.execute(st)
        check(st.get_state(), ref, n, dtype)
        plan.execute(st)  # again, on its own output
        check(st.get_state(), ref2, n, dtype)
        st.set_state(psi0)
        plan.execute_range(st, 0, 1)  # the passes stay there, one by one
        plan.execute_range(st, 1, plan.info["passes"] - 1)
        check(st.get_state(), ref, n, dtype)
        plan.execute_from_basis(st, x)
        check(st.get_state(), base, n, dtype)
        st.set_state(psi0)
        st.run(c, mode=mode, max_fused=4)  # one-shot: no operands of the passes
        check(st.get_state(), ref, n, dtype)


@pytest.mark.parametrize("dtype", [C64, C128])
def test_program_cuts(qsim, dtype):
    """A narrow state whose gates all share one tile: the program is cut where its shared memory ends."""
    n = 6
    rng = np.random.default_rng(11)
    c = W.Circuit(n)
    for i in range(700):
        a, b = (int(x) for x in rng.permutation(n)[:2])
        c.append(W.Gate((a, b), (), W.haar_unitary(4, rng), "u4"))
    psi0 = random_state(n, 5)
    psi0 = psi0.astype(np.complex64) if dtype == C64 else psi0
    ref = oracle.run(c, psi=psi0.astype(np.complex128))
    for mode in (0, 1):
        st = qsim.State(n, dtype)
        st.set_state(psi0)
        st.run(c, mode=mode, max_fused=4)
        check(st.get_state(), ref, n, dtype)
