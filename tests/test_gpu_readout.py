"""Readout kernels at the widths where their paths change, against the FP64 oracle.

Sums of |a|^2 are float-float (relative error below 2^-44 of the total here, taken as 1e-13); indices of samples are
equal.
"""
import numpy as np
import pytest

import oracle
from helpers import random_state

pytestmark = pytest.mark.gpu

C64, C128 = 0, 1


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


def state(qsim, n, dtype, seed):
    psi = random_state(n, seed)
    psi = psi.astype(np.complex64) if dtype == C64 else psi
    st = qsim.State(n, dtype)
    st.set_state(psi)
    return st, psi.astype(np.complex128)


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n", [1, 2, 11, 12, 13, 14, 17])
def test_pauli_strings(qsim, dtype, n):
    """Z alone, flips of qubit 0 alone, with and without qubit 0, an even and an odd number of Y, top and low flips:
    the wide kernels start at 12 (no flips) and 13 qubits."""
    st, psi = state(qsim, n, dtype, n)
    rng = np.random.default_rng(n)
    strings = ["I" * n, "Z" * n, "X" + "I" * (n - 1), "Y" + "Z" * (n - 1), "I" * (n - 1) + "X", "I" * (n - 1) + "Y",
               "X" * n, "Y" * n, "I" * (n // 2) + "Y" * (n - n // 2)]
    strings += ["".join(rng.choice(list("IXYZ"), n)) for _ in range(6)]
    for p in strings:
        assert abs(st.expect_pauli(p) - oracle.expect_pauli(psi, n, p)) <= 1e-13, p
    assert abs(st.norm() - oracle.norm2(psi, n)) <= 1e-13


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n", [1, 3, 5, 6, 8, 12, 13, 18, 22])
def test_samples(qsim, dtype, n):
    """Segments of 2^n to 2^12 amplitudes, one to many segments and chunks; alone and after the <Z> statistics."""
    st, psi = state(qsim, n, dtype, n + 50)
    u = oracle.uniforms(77, 500)
    want = oracle.sample(psi, n, u)
    assert np.array_equal(st.sample_uniforms(u), want)
    assert np.array_equal(st.sample(77, 500), want)
    zi, zz, got = st.expect_z_and_sample(77, 500)
    assert np.array_equal(got, want)
    z2, zz2 = st.expect_z()
    assert np.array_equal(zi, z2) and np.array_equal(zz, zz2)
    assert np.array_equal(st.sample(77, 5000)[:500], want)  # more than the pinned buffer holds


@pytest.mark.parametrize("dtype", [C64, C128])
def test_samples_of_sparse_states(qsim, dtype):
    """Amplitudes of zero are never drawn, nor segments or chunks without weight, at either end of the interval."""
    n = 22
    psi = np.zeros(1 << n, dtype=np.complex64 if dtype == C64 else np.complex128)
    at = np.array([5, 4095, 4096, 1 << 20, (1 << 21) + 77, (1 << n) - 3])
    psi[at] = np.sqrt(np.array([0.25, 0.25, 0.125, 0.125, 0.125, 0.125]))
    st = qsim.State(n, dtype)
    st.set_state(psi)
    # (between the steps of the distribution: at one, rounding of the weights decides)
    u = np.concatenate([[0.0, np.nextafter(1.0, 0.0)], (np.arange(200) + 0.5) / 200])
    got = st.sample_uniforms(u)
    assert np.array_equal(got, oracle.sample(psi.astype(np.complex128), n, u))


@pytest.mark.parametrize("dtype", [C64, C128])
@pytest.mark.parametrize("n,qubits", [(12, (3,)), (20, (0, 19)), (22, (1,)), (22, (21, 10, 9)), (16, tuple(range(12)))])
def test_marginals(qsim, dtype, n, qubits):
    """Few bins with many partial sums and many bins with few."""
    st, psi = state(qsim, n, dtype, n + 9)
    assert np.max(np.abs(st.probs(qubits) - oracle.probs(psi, n, qubits))) <= 1e-13


@pytest.mark.parametrize("scale", [1.0, 1e-15, 1e15])
def test_complex128_magnitudes(qsim, scale):
    """Double-precision amplitudes reach the float-float sums by integer splitting: over the magnitudes whose squares
    a float holds with its remainder, the sums scale exactly; smaller ones vanish."""
    n = 13
    psi = random_state(n, 4) * scale
    psi[7] = 1e-200
    psi[9] = 5e-324
    st = qsim.State(n, C128)
    st.set_state(psi)
    want = oracle.norm2(psi, n)
    assert abs(st.norm() - want) <= 1e-13 * want
    assert np.max(np.abs(st.probs([0, 12]) - oracle.probs(psi, n, [0, 12]))) <= 1e-13 * want
    psi[3] = np.inf
    st.set_state(psi)
    assert not np.isfinite(st.norm())
