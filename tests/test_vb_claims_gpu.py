"""Claimed slices (grid-wide sweeps of four replicas, and of two where the spins lie far beyond L2) against the
oracle: classes of just fewer and just more slices than are claimed from, several classes of either kind,
batches, calls of one sweep and of several, and a handle that goes on after another one of its size.
Spins equal."""
import numpy as np
import pytest

import oracle
import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TEMPS = [1.0, 0.6, 3.0, 0.0]


@pytest.fixture(scope="module")
def sg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as m
    return m


def run_and_compare(sg, graphs, R, calls, lanes):
    insts = []
    for b, (rp, col, eid) in enumerate(graphs):
        jb = sg_inputs.vb_lane_couplings(eid, int(eid.max()) + 1 if eid.size else 0, 5 + b)
        insts.append(dict(row_ptr=rp, col=col, jbits=jb, seed=(9 << 33) + b, temps=TEMPS[:R]))
    run = sg.VBRun(insts, n_lanes=64, n_replicas=R)
    for n in calls:
        run.sweep(n)
    run.synchronize()
    spins = run.spins()
    run.close()
    mask = np.uint64((1 << lanes) - 1)
    for g, s in zip(insts, spins):
        ref = oracle.vb_run(g["row_ptr"], g["col"], g["jbits"], lanes, g["temps"], g["seed"], sum(calls), [], [])
        assert np.array_equal(s & mask, ref["spins"] & mask)


# 304 CTAs of 6 warps: classes of more than 3656 slices are claimed from (bipartite: N / 64 slices each)
@pytest.mark.parametrize("n", [2 * 32 * 3655, 2 * 32 * 3656, 2 * 32 * 3657, 2 * 32 * 3664, 600_002])
def test_two_classes(sg, n):
    run_and_compare(sg, [sg_inputs.random_regular_graph(n, 3, 1, bipartite=True)], 4, [1, 4, 3], 1)


@pytest.mark.parametrize("n,c", [(450_001, 4.0), (900_000, 3.0), (700_000, 9.0), (500_000, 0.01)])
def test_several_classes(sg, n, c):
    run_and_compare(sg, [sg_inputs.poisson_graph(n, c, 2)], 4, [2, 1, 4], 1)


def test_batch(sg):
    graphs = [sg_inputs.poisson_graph(n, 4.0, b) for b, n in enumerate([300_000, 40, 500_001, 2000])]
    run_and_compare(sg, graphs, 4, [3, 2], 1)


def test_two_replicas_far_beyond_l2(sg):
    run_and_compare(sg, [sg_inputs.poisson_graph(12_000_001, 1.0, 3)], 2, [1, 3], 1)
