"""The configuration read back: more words than one part of the packed read-back, uneven graphs, and SK
sizes that are no multiple of the four spins a thread writes, against the oracle's spins."""
import numpy as np
import pytest

import oracle
import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_configuration_read_back_in_parts():
    """More words than one part of the read-back: the initial spins of 2^21 + 5 vertices, 4 replicas."""
    n = (1 << 21) + 5
    i = np.arange(n - 1)
    rp = np.zeros(n + 1, dtype=np.int32)
    rp[1:] = np.cumsum(np.where((np.arange(n) == 0) | (np.arange(n) == n - 1), 1, 2))
    col = np.empty(2 * (n - 1), dtype=np.int32)
    col[rp[:-1][1:]] = i            # the neighbour before
    col[rp[1:][:-1] - 1] = i + 1    # the neighbour after
    import paper_1906_11195_gb300 as sg
    jb = np.zeros(col.size, dtype=np.uint64)
    run = sg.VBRun([dict(row_ptr=rp, col=col, jbits=jb, seed=4, temps=[1.0] * 4)], n_replicas=4)
    got = run.spins()[0]
    run.close()
    ref = oracle.vb_run(rp, col, jb, 2, [1.0] * 4, 4, 0, [], [])["spins"]
    assert np.array_equal(got & np.uint64(3), ref & np.uint64(3))


@pytest.mark.parametrize("n", [2, 129, 1001, 1002, 1003])
def test_sk_spins(n):
    import paper_1906_11195_gb300 as sg
    J = sg_inputs.sk_couplings(n, n)
    temps = [0.5] * 32
    run = sg.SKRun(J, temps, 6)
    run.sweep(2)
    got = run.spins()
    run.close()
    assert np.array_equal(got, oracle.sk_run(J, temps, 6, 2, [], [])["spins"])
