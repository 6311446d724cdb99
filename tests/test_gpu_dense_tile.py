"""Dense 5- and 6-qubit passes at every number of groups a CTA takes (1, 4, 16, 64), with and without controls, against
the FP64 oracle; complex64 max |amplitude error| <= 1e-5, complex128 <= 1e-12, as for the other passes."""
import numpy as np
import pytest

import oracle
import workloads as W
from helpers import random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("n", [5, 6, 7, 10, 13, 14, 15, 16, 17, 18, 19, 20])
def test_groups_per_cta(qsim, dtype, k, n):
    if n < k:
        return
    rng = np.random.default_rng(100 * k + n)
    c = W.Circuit(n)
    for nc in (0, min(2, n - k)):
        q = [int(x) for x in rng.permutation(n)]
        c.append(W.Gate(tuple(q[:k]), tuple(q[k:k + nc]), W.haar_unitary(1 << k, rng), "u"))
    p = qsim.Plan(c, dtype, mode=0, launch_per_pass=True)
    assert all(x["kind"] == "dense_tile" for x in p.passes())
    psi = random_state(n, 7)
    psi = psi.astype(np.complex64) if dtype == 0 else psi
    st = qsim.State(n, dtype)
    st.set_state(psi)
    p.execute(st)
    err = np.max(np.abs(st.get_state().astype(np.complex128) - oracle.run(c, psi=psi.astype(np.complex128))))
    assert err <= (1e-5 if dtype == 0 else 1e-12)
