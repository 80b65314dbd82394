"""The packed measurement launch (C of every snapshot, q and E at once) at the sizes where its split
can go wrong: one slice, runs that end inside a CTA, batches whose CTAs hold several graphs and come
back to the first one in the next colour class, every replica count.  Counts are integers: equal."""
import numpy as np
import pytest

import oracle
import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def instance(n, c, seed, temps):
    rp, col, eid = sg_inputs.poisson_graph(n, c, seed)
    jb = sg_inputs.vb_lane_couplings(eid, eid.max() + 1 if eid.size else 0, seed)
    return dict(row_ptr=rp, col=col, jbits=jb, seed=seed, temps=temps)


@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("sizes,c", [([2], 1.0), ([33], 4.0), ([8000], 4.0), ([20011], 5.0),
                                     ([300, 300, 300], 4.0), ([40, 700, 64, 900, 33, 500], 4.0),
                                     ([5000, 17, 5000], 3.0)])
def test_measurement_matches_oracle(R, sizes, c):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_11195_gb300 as sg
    temps = [1.0, 0.6, 0.8, 1.2][:R]
    graphs = [instance(n, c, 50 + i, temps) for i, n in enumerate(sizes)]
    tw, tm = [0, 1, 3], [0, 1, 2, 3, 5]
    run = sg.VBRun(graphs, n_lanes=64, n_replicas=R, tw=tw, tm=tm)
    run.sweep(5)
    C, q, E = run.results()
    now = run.measure()
    run.close()
    for b, g in enumerate(graphs):
        ref = oracle.vb_run(g["row_ptr"], g["col"], g["jbits"], 64, g["temps"], g["seed"], 5, tw, tm)
        assert np.array_equal(C[b], ref["C"]) and np.array_equal(E[b], ref["E"])
        assert np.array_equal(q[b], ref["q"])
        assert np.array_equal(now[0][b], ref["C"][..., -1]) and np.array_equal(now[2][b], ref["E"][..., -1])
