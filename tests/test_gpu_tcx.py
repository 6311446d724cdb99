"""Blocks of up to 5 qubits in the state's own precision on the tensor cores (exact integer slices), against the
FP64 oracle.

Tolerance: the fixed-point steps of the row and of U and the final rounding leave at most a few units of
2^-53 (complex128) or 2^-24 (complex64) of the row's largest amplitude per block; composing the block in FP64 adds
its own roundings. Bound per block: 32 * 2^-53 and 4 * 2^-24 of the state's largest amplitude.
"""
import numpy as np
import pytest

import oracle
import workloads as W
from helpers import random_state

pytestmark = pytest.mark.gpu

C64, C128 = 0, 1
EPS = {C64: 4 * 2.0 ** -24, C128: 32 * 2.0 ** -53}


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


def block(n, qubits, seed):
    """Gates that fuse into one dense block on `qubits`."""
    rng = np.random.default_rng(seed)
    c = W.Circuit(n)
    for q in qubits:
        c.append(W.Gate((q,), (), W.haar_unitary(2, rng), "u"))
    for a, b in zip(qubits, qubits[1:]):
        c.append(W.Gate((b,), (a,), W.haar_unitary(2, rng), "cu"))
    c.append(W.Gate((qubits[0],), (), W.haar_unitary(2, rng), "u"))
    return c


def run(qsim, c, dtype, psi0=None, basis=None):
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


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n,qubits", [
    (17, (0, 1, 2, 3, 4)), (17, (12, 13, 14, 15, 16)), (17, (0, 3, 7, 11, 16)), (18, (1, 2, 3, 4, 5)),
    (18, (0, 1, 5, 9, 17)), (19, (7, 8, 9, 10)), (20, (0, 2)), (20, (19,)), (20, (0,)), (21, (5, 6, 7, 8, 9)),
    (21, (0, 1, 2)), (22, (0, 5, 10, 15, 21))])
def test_block_against_oracle(qsim, dtype, n, qubits):
    """Low, high and scattered windows, padded blocks of 1..4 qubits, one to several tiles per CTA."""
    c = block(n, qubits, seed=n + sum(qubits))
    psi0 = random_state(n, n)
    g = run(qsim, c, dtype, psi0.astype(np.complex64) if dtype == C64 else psi0)
    ref = oracle.run(c, psi=(psi0.astype(np.complex64) if dtype == C64 else psi0).astype(np.complex128))
    assert np.max(np.abs(g - ref)) <= EPS[dtype] * np.max(np.abs(psi0))


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("x", [0, 1, 0b10110011100011110])
def test_from_basis(qsim, dtype, x):
    c = block(17, (2, 4, 6, 8, 16), seed=3)
    assert np.max(np.abs(run(qsim, c, dtype, basis=x) - oracle.run(c, basis_state=x))) <= EPS[dtype]


@pytest.mark.parametrize("dtype,scale", [(C64, 2.0 ** -120), (C64, 2.0 ** 90), (C128, 2.0 ** -1000), (C128, 2.0 ** 900)])
def test_scales(qsim, dtype, scale):
    """Rows near both ends of the exponent range, and rows of zeros."""
    n, c = 17, block(17, (0, 4, 8, 12, 16), seed=4)
    dt = np.complex64 if dtype == C64 else np.complex128
    psi0 = random_state(n, 5).astype(dt)
    psi0[: 1 << 15] = 0
    out = run(qsim, c, dtype, (psi0 * dt(scale)).astype(dt))
    ref = oracle.run(c, psi=psi0.astype(np.complex128))
    tiny = np.finfo(np.float32 if dtype == C64 else np.float64).tiny
    back = out.astype(np.complex128) / scale
    assert np.max(np.abs(back - ref)) <= EPS[dtype] * np.max(np.abs(psi0)) + 4 * tiny / scale


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinity_and_nan_stay_in_their_rows(qsim, dtype, value):
    """A row with a non-finite amplitude becomes NaN; every other row keeps its values."""
    n, qubits = 17, (1, 4, 8, 12, 16)
    c = block(n, qubits, seed=6)
    psi0 = random_state(n, 7).astype(np.complex64 if dtype == C64 else np.complex128)
    good = run(qsim, c, dtype, psi0)
    at = 0b01011001110010110
    psi0[at] = value
    out = run(qsim, c, dtype, psi0)
    mask = sum(1 << q for q in qubits)
    row = (np.arange(1 << n) & ~mask) == (at & ~mask)
    assert np.all(np.isnan(out[row].real) & np.isnan(out[row].imag))
    assert np.array_equal(out[~row], good[~row])


@pytest.mark.parametrize("dtype", [C64, C128])
def test_exact_products(qsim, dtype):
    """Digits at their limits: the sums of products stay exact integers, so a uniform state through Hadamards and
    a permutation gives its exact values, and the inverse block gives the input back."""
    n, qubits = 18, (0, 3, 6, 9, 12)
    c = W.Circuit(n)
    for q in qubits:
        c.append(W.Gate((q,), (), W.H(), "h"))
    c.append(W.Gate((0,), (3,), W.X(), "cx"))
    dt = np.complex64 if dtype == C64 else np.complex128
    a = np.nextafter(np.float32(1), np.float32(0)) if dtype == C64 else np.nextafter(1.0, 0.0)
    psi0 = np.full(1 << n, (a + 1j * a), dtype=dt)
    out = run(qsim, c, dtype, psi0)
    ref = oracle.run(c, psi=psi0.astype(np.complex128))
    assert np.max(np.abs(out - ref)) <= EPS[dtype] * np.max(np.abs(ref))
