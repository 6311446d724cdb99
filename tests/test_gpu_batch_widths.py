"""Batched circuits of 1 to 18 qubits at every fusion width: passes of few groups (several lanes a group), one group a
thread and two, in shared memory and in clusters, against the FP64 oracle; <Z_i> and <Z_i Z_{i+1}> within 1e-5, as for
the other batched circuits."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_every_width(qsim, k):
    rng = np.random.default_rng(50 + k)
    cs = [W.Circuit(1), W.Circuit(7), W.Circuit(15)]  # no gates
    for n in range(1, 19):
        c = W.Circuit(n)
        for _ in range(30):
            q = [int(x) for x in rng.permutation(n)[:min(n, k)]]
            if len(q) > 1 and rng.random() < 0.4:
                c.append(W.Gate((q[0], q[1]), (), W.haar_unitary(4, rng), "u4"))
            else:
                c.append(W.Gate((q[0],), (), W.haar_unitary(2, rng), "u"))
        cs.append(c)
    b = qsim.Batch(cs, max_fused=k)
    b.execute()
    for (zi, zz), c in zip(b.results(), cs):
        rzi, rzz = oracle.expect_z_chain(oracle.run(c), c.n)
        np.testing.assert_allclose(zi, rzi, atol=1e-5, rtol=0)
        np.testing.assert_allclose(zz, rzz, atol=1e-5, rtol=0)
