"""Batched circuits wide enough to run as plans in the states' own precision (from 19 qubits on, no fusion width
given) against the FP64 oracle: <Z_i> and <Z_i Z_{i+1}> within 1e-5, as for the other batched circuits."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsim(gpu_lib):
    from paper_2511_14664_gb300 import qsim as q
    return q


def circuits():
    """Both sides of the width, an empty circuit, general gates on 1 to 4 qubits, chains."""
    rng = np.random.default_rng(31)
    cs = [W.Circuit(19)]
    for n in (18, 19, 21):
        c = W.Circuit(n)
        for _ in range(50):
            c.append(W.random_gate(n, rng, kmax=2, cmax=2, diag_prob=0.3))
        c.append(W.Gate((3, n - 1, 0, 7), (), W.haar_unitary(16, rng), "u4"))
        cs.append(c)
    return cs + [W.tfim_chain(n, s, 0.4, 0.9) for n, s in ((12, 3), (18, 4), (19, 6), (20, 4), (22, 3))]


def check(results, refs):
    for (zi, zz), (rzi, rzz) in zip(results, refs):
        np.testing.assert_allclose(zi, rzi, atol=1e-5, rtol=0)
        np.testing.assert_allclose(zz, rzz, atol=1e-5, rtol=0)


@pytest.mark.parametrize("prec,tc_min_n", [(0, 0), (4, 21), (1, 26)])
def test_against_oracle(qsim, prec, tc_min_n):
    cs = circuits()
    refs = [oracle.expect_z_chain(oracle.run(c), c.n) for c in cs]
    b = qsim.Batch(cs, precision=prec, tc_min_n=tc_min_n)
    assert b.ws_bytes == 8 * sum(2 ** c.n for c in cs if c.n > 13)
    assert (b.info["tc_blocks"] > 0) == (prec != 0 and tc_min_n <= 22)
    b.execute()
    r1 = b.results()
    check(r1, refs)
    b.execute(use_graph=True)
    b.execute(use_graph=True)
    r2 = b.results()
    r3, _ = qsim.batch_run(cs, precision=prec, tc_min_n=tc_min_n)
    for (a1, b1), (a2, b2), (a3, b3) in zip(r1, r2, r3):
        assert np.array_equal(a1, a2) and np.array_equal(b1, b2)
        assert np.array_equal(a1, a3) and np.array_equal(b1, b3)
