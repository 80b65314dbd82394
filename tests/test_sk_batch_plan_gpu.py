"""Persistent SK launches planned side by side: samples of one batch with different splits, and handles
whose launches need less shared memory prepared between a handle's preparation and its first sweep."""
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


@pytest.mark.parametrize("R,sizes", [(32, [1500, 700, 2100]), (128, [640, 1700, 900, 1300, 2500]),
                                     (64, [1000] * 9)])
def test_batch_matches_oracle(R, sizes):
    import paper_1906_11195_gb300 as sg
    samples = [dict(J=sg_inputs.sk_couplings(n, 30 + i), seed=90 + i, temps=[0.4] * (R // 2) + [0.9] * (R // 2))
               for i, n in enumerate(sizes)]
    run = sg.SKBatchRun(samples, R, block=128, tw=[0], tm=[])
    run.sweep(5)
    run.synchronize()
    spins = run.spins()
    run.close()
    for s, x in zip(spins, samples):
        assert np.array_equal(s, oracle.sk_run(x["J"], x["temps"], x["seed"], 5, [], [])["spins"])


def test_handles_prepared_in_turn():
    import paper_1906_11195_gb300 as sg
    n = 1100
    J = sg_inputs.sk_couplings(n, 8)
    temps = {R: [0.5] * R for R in (256, 128, 32)}
    runs = {R: sg.SKRun(J, temps[R], 4, block=128) for R in temps}
    for R, run in runs.items():
        run.sweep(3)
        run.synchronize()
        got = run.spins()
        run.close()
        assert np.array_equal(got[:8], oracle.sk_run(J, temps[R][:8], 4, 3, [], [])["spins"])
