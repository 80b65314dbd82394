"""The packed sweep's forms against the oracle where each can go wrong: one CTA's shared memory (a
single slice; classes of more slices than warps), clusters of 2 to 16 CTAs (more and fewer slices
than CTAs; several graphs, one cluster each, one graph without vertices in the last classes), the
grid-wide form with chunks of 8 and of 4 entries, the thin last classes, slices wider than the
four-plane counter, and batches with more graphs than threshold tables in shared memory.  Sweeps are
taken in uneven calls.  Integers: equal."""
import numpy as np
import pytest

import oracle
import sg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TEMPS = [1.0, 0.6, 3.0, 0.0]


def poisson(n, c, seed):
    return sg_inputs.poisson_graph(n, c, seed)


def hubs(n, degrees, seed):
    """Vertices 0, 1, ... of the given degrees, joined to the vertices after them, and a path."""
    rng = np.random.default_rng(seed)
    edges = {(i, i + 1) for i in range(len(degrees), n - 1)}
    for h, d in enumerate(degrees):
        edges |= {(h, int(j)) for j in rng.choice(np.arange(len(degrees), n), d, replace=False)}
    lo, hi = (np.array(x, dtype=np.int64) for x in zip(*sorted(edges)))
    src, dst, eid = np.concatenate([lo, hi]), np.concatenate([hi, lo]), np.tile(np.arange(lo.size), 2)
    order = np.lexsort((dst, src))
    rp = np.zeros(n + 1, dtype=np.int32)
    rp[1:] = np.cumsum(np.bincount(src, minlength=n))
    return rp, dst[order].astype(np.int32), eid[order]


def run_and_compare(graphs, R, sweeps, lanes, chunks):
    import paper_1906_11195_gb300 as sg
    insts = []
    for b, (rp, col, eid) in enumerate(graphs):
        jb = sg_inputs.vb_lane_couplings(eid, int(eid.max()) + 1 if eid.size else 0, 7 + b)
        insts.append(dict(row_ptr=rp, col=col, jbits=jb, seed=(11 << 33) + b, temps=TEMPS[:R]))
    run = sg.VBRun(insts, n_lanes=64, n_replicas=R)
    for c in chunks:
        run.sweep(c)
    run.sweep(sweeps - sum(chunks))
    run.synchronize()
    spins = run.spins()
    run.close()
    mask = np.uint64(0xFFFFFFFFFFFFFFFF) if lanes == 64 else np.uint64((1 << lanes) - 1)
    for b, g in enumerate(insts):
        ref = oracle.vb_run(g["row_ptr"], g["col"], g["jbits"], lanes, g["temps"], g["seed"], sweeps, [], [])
        assert np.array_equal(spins[b] & mask, ref["spins"] & mask)


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("n", [2, 31, 33, 700, 1300, 2500, 9000, 24000, 40001])
def test_one_graph(n, R):
    run_and_compare([poisson(n, 1.0 if n == 2 else 4.0, n)], R, 9, 64 if n < 3000 else 5, [1, 5])


@pytest.mark.parametrize("n,R", [(250_001, 1), (250_001, 2), (190_000, 4)])
def test_more_slices_than_warps(n, R):
    run_and_compare([poisson(n, 4.0, 3)], R, 4, 2, [1])


@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("n", [200, 9000, 60000])
def test_wide_slices(n, R):
    run_and_compare([hubs(n, [63, 16, 15, 33, 8], 5)], R, 6, 8, [2])


@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("sizes", [[40, 700, 64, 900, 33], [3000, 5000, 100, 2], [600] * 20,
                                   [3000] * 20, [70000, 50, 3000], [1200] * 17 + [30000]])
def test_batches(sizes, R):
    graphs = [poisson(n, 1.0 if n == 2 else 4.0 if b % 2 else 3.0, b) for b, n in enumerate(sizes)]
    run_and_compare(graphs, R, 5, 3, [2])
