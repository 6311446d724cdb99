"""The phase pass at every split of the index bits (1 to 16 ranges a warp, 1 to 8 warps a block), launched by itself,
against the product of the same diagonal gates in 64 bits; tolerances as for the other phase passes (complex64 max
|amplitude error| <= 1e-5, complex128 <= 1e-12)."""
import numpy as np
import pytest

import workloads as W
from helpers import random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [10, 11, 14, 17, 18, 20, 21, 22, 23, 24])
@pytest.mark.parametrize("joined", [True, False])
def test_widths(qsim, dtype, n, joined):
    """joined: terms between index bits 0..4 and 5..9."""
    rng = np.random.default_rng(n)
    c = W.Circuit(n)
    phase = np.zeros(1 << n)
    x = np.arange(1 << n)
    for a, b in [(0, n - 1), (3, 7), (5, 9), (4, 8), (1, 2), (n - 2, n - 1), (6, n - 3)] + \
            [tuple(int(q) for q in rng.permutation(n)[:2]) for _ in range(12)]:
        th = float(rng.uniform(0, 6))
        if not joined and min(a, b) < 5 <= max(a, b) < 10:
            continue
        c.append(W.Gate((a,), (b,), W.CP(th), "cp"))
        phase += th * ((x >> a) & (x >> b) & 1)
    p = qsim.Plan(c, dtype, mode=1, max_fused=5, launch_per_pass=True)
    assert [q["kind"] for q in p.passes()] == ["phase"]
    psi = random_state(n, 3)
    psi = psi.astype(np.complex64) if dtype == 0 else psi
    st = qsim.State(n, dtype)
    st.set_state(psi)
    p.execute(st)
    err = np.max(np.abs(st.get_state().astype(np.complex128) - psi * np.exp(1j * phase)))
    assert err <= (1e-5 if dtype == 0 else 1e-12)
