"""Batches at the number of graphs whose thresholds the grid-wide sweep keeps in shared memory (32) and just
beyond it, where it reads them from global memory: one slice a warp (chunks of 8), several (chunks of
4) and, with four replicas, claimed slices.  Spins equal the oracle's."""
import numpy as np
import pytest

import oracle
import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TEMPS = [1.0, 0.6, np.inf, 0.0]  # at infinite temperature every draw passes the first thresholds


@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("small,large", [(31, 30000), (32, 30000), (32, 260_000), (70, 9000)])
def test_spins(small, large, R):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as sg
    graphs = []
    for b, n in enumerate([1200] * small + [large]):
        rp, col, eid = sg_inputs.poisson_graph(n, 4.0, b)
        jb = sg_inputs.vb_lane_couplings(eid, int(eid.max()) + 1, b)
        temps = (TEMPS[b % 4:] + TEMPS[:b % 4])[:R]
        graphs.append(dict(row_ptr=rp, col=col, jbits=jb, seed=(3 << 32) + b, temps=temps))
    run = sg.VBRun(graphs, n_lanes=64, n_replicas=R)
    run.sweep(1)
    run.sweep(3)
    run.synchronize()
    spins = run.spins()
    run.close()
    for g, s in zip(graphs, spins):
        ref = oracle.vb_run(g["row_ptr"], g["col"], g["jbits"], 3, g["temps"], g["seed"], 4, [], [])
        assert np.array_equal(s & np.uint64(7), ref["spins"] & np.uint64(7))
