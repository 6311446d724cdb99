"""Blocks of up to 5 qubits in the state's own precision: amplitudes and matrix entries that are small beside others keep
their digits.

Tolerance, for every amplitude y_r = sum_c U_rc x_c by itself: the slices' error is below 2^-25 (complex64) or 2^-52
(complex128) of the power of two above a row's largest amplitude, and they take only rows in which sum_c |U_rc| |x_c| is
above 2^-9 of that for every r. Other rows are sums of FMA chains, at most 64 * 2^-24 (2^-53) of that sum, and U itself is
rounded once. Both: 2^-16 (2^-43) of the sum.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

C64, C128 = 0, 1
DT = {C64: np.complex64, C128: np.complex128}
TOL = {C64: 2.0 ** -16, C128: 2.0 ** -43}


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


def run(qsim, c, dtype, psi0=None, basis=0):
    p = qsim.Plan(c, dtype, mode=1, max_fused=5)
    assert p.info["passes"] == 1
    st = qsim.State(c.n, dtype)
    if psi0 is None:
        p.execute_from_basis(st, basis)
    else:
        st.set_state(psi0)
        p.execute(st)
    st.synchronize()
    return st.get_state()


def matrix(c, qubits):
    """The block's matrix on `qubits` (ascending), column by column."""
    at = {q: j for j, q in enumerate(qubits)}
    s = W.Circuit(len(qubits))
    for g in c.gates:
        s.append(W.Gate(tuple(at[q] for q in g.targets), tuple(at[q] for q in g.controls), g.matrix, g.name))
    return np.stack([oracle.run(s, basis_state=x) for x in range(1 << len(qubits))], axis=1)


def rows(v, n, qubits):
    """v with the block's amplitudes along the last axis (bit j of it <-> qubits[j])."""
    axes = [n - 1 - q for q in range(n) if q not in qubits] + [n - 1 - q for q in reversed(qubits)]
    return v.reshape((2,) * n).transpose(axes).reshape(-1, 1 << len(qubits))


def circuit(n, qubits, kind, seed):
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    if kind == "turn":      # close to the identity: products of small sines
        for q in qubits:
            c.append(W.Gate((q,), (), W.RY(0.02), "ry"))
        return c
    for q in qubits:
        c.append(W.Gate((q,), (), W.haar_unitary(2, rng), "u"))
    for a, b in zip(qubits, qubits[1:]):
        c.append(W.Gate((b,), (a,), W.haar_unitary(2, rng), "cu"))
    return c


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("theta", [2e-4, 0.2, 2.0])
def test_small_rotations_of_a_basis_state(qsim, dtype, theta):
    """R_y on five qubits of |0...0>: the amplitude with j flips is sin^j cos^(5-j), down to 1e-20."""
    n, qubits = 17, (3, 5, 8, 12, 16)
    c = W.Circuit(n)
    for q in qubits:
        c.append(W.Gate((q,), (), W.RY(theta), "ry"))
    out = rows(run(qsim, c, dtype).astype(np.complex128), n, qubits)
    flips = np.array([bin(m).count("1") for m in range(32)])
    ref = np.sin(theta / 2) ** flips * np.cos(theta / 2) ** (5 - flips)
    assert np.all(np.abs(out[0] - ref) <= TOL[dtype] * np.abs(ref))
    assert not np.any(out[1:])


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("spread", [4, 8, 14, 40])
@pytest.mark.parametrize("kind", ["dense", "turn"])
@pytest.mark.parametrize("n,qubits", [(17, (0, 1, 2, 3, 4)), (17, (2, 6, 9, 13, 16)), (20, (0, 3, 7, 11, 19)),
                                      (21, (8, 9, 10, 11)), (20, (0, 5, 12)), (20, (4, 19)), (20, (7,))])
def test_rows_of_wide_range(qsim, dtype, spread, kind, n, qubits):
    """Amplitudes spread over up to 40 binades, some of them zero; whole rows of even size among them; blocks padded with
    idle qubits (1 to 4 qubits)."""
    rng = np.random.default_rng(n + spread + sum(qubits))
    psi0 = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    size = np.exp2(-rng.uniform(0, spread, 1 << n))
    size[rng.random(1 << n) < 0.05] = 0
    size[: 1 << (n - 2)] = 1            # rows that the slices take, beside the others
    size[1 << (n - 1): 3 << (n - 2)] *= np.exp2(-20.0)
    psi0 = (psi0 * size).astype(DT[dtype])
    c = circuit(n, qubits, kind, seed=spread)
    some = rng.integers(0, 1 << (n - len(qubits)), 1500)
    out = rows(run(qsim, c, dtype, psi0), n, qubits)[some].astype(np.clongdouble)
    U, x = matrix(c, qubits).astype(np.clongdouble), rows(psi0, n, qubits)[some].astype(np.clongdouble)
    ref = x @ U.T
    total = (np.abs(x) @ np.abs(U).T).astype(np.float64)
    assert np.all(np.abs(out - ref).astype(np.float64) <= TOL[dtype] * total + np.finfo(np.float32).tiny * (dtype == C64))


@pytest.mark.parametrize("dtype,n,qubits", [(C64, 20, (2, 6, 11, 17)), (C128, 20, (2, 6, 11, 17)), (C128, 18, (0, 5, 12)),
                                            (C128, 20, (4, 19)), (C128, 21, (7,))])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_amplitudes_stay_in_their_groups(qsim, dtype, n, qubits, value):
    """Blocks padded with idle qubits: only the amplitudes that the block joins with a non-finite one become so."""
    rng = np.random.default_rng(n)
    psi0 = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)).astype(DT[dtype])
    c = circuit(n, qubits, "dense", seed=3)
    good = run(qsim, c, dtype, psi0)
    at = 0b101100111001011001101 & ((1 << n) - 1)
    psi0[at] = value
    out = run(qsim, c, dtype, psi0)
    mask = sum(1 << q for q in qubits)
    group = (np.arange(1 << n) & ~mask) == (at & ~mask)
    assert np.count_nonzero(group) == 1 << len(qubits)
    assert not np.any(np.isfinite(out[group]))
    assert np.max(np.abs(out[~group] - good[~group])) <= 2 * TOL[dtype] * np.max(np.abs(good[~group]))


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n,qubits", [(17, (1, 4, 8, 12, 16)), (18, (0, 1, 2, 3, 4)), (20, (3, 9, 15))])
def test_sparse_blocks_of_sparse_states(qsim, dtype, n, qubits):
    """Controlled-NOTs and half turns, whose products have exact zeros, on states of few amplitudes: results to which
    nothing adds are zero, the others keep their digits."""
    half = 0.5 * np.array([[1 + 1j, 1 - 1j], [1 - 1j, 1 + 1j]])
    c = W.Circuit(n)
    for a, b in zip(qubits, qubits[1:]):
        c.append(W.Gate((b,), (a,), W.X(), "cx"))
    for q in qubits[::2]:
        c.append(W.Gate((q,), (), half, "sx"))
    c.append(W.Gate((qubits[0],), (qubits[-1],), W.X(), "cx"))
    rng = np.random.default_rng(n)
    psi0 = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi0 *= (rng.random(1 << n) < 0.1) * np.exp2(-rng.uniform(0, 3, 1 << n))
    psi0[::7] *= 2.0 ** -15
    psi0 = psi0.astype(DT[dtype])
    out = rows(run(qsim, c, dtype, psi0), n, qubits)
    U, x = matrix(c, qubits), rows(psi0.astype(np.complex128), n, qubits)
    total = np.abs(x) @ np.abs(U).T
    assert np.any(total == 0)
    assert np.all(np.abs(out - x @ U.T) <= TOL[dtype] * total)
