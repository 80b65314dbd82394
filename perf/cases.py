"""The work that users of this library have it do, as cases of stated sizes.

A program that studies aging creates an instance (a Viana-Bray graph with 64 coupling sets, a
batch of graphs, an SK sample or a batch of them), lets it run for some sweeps, and looks at the
correlation with its snapshots, the replica overlap and the energy; then it runs on.  Most cases
here are one such step on an instance that is already set up: `run` advances the state and returns
what the measurement gives, for every lane, replica and snapshot.  Where `spins` is set the program
also reads the configuration back, as it does for small instances and now and then for larger
ones.  The others are a whole quench from the host arrays to its results, a run measured at every
sweep, and the SK fields of a caller that owns all its memory.

Every result is an integer count, the same for every correct implementation.
"""
import math

import numpy as np
import torch

import paper_1906_11195_gb300 as sg
import sg_inputs

T_08_TC = 0.8 / math.atanh(1.0 / math.sqrt(3.0))  # 0.8 T_c of the random regular graph, degree 4


def listed():
    return [
        # one small Poissonian graph, the lower end of the uneven batch's sizes and the size of the
        # first aging runs: a sweep is a few microseconds of work, launches and barriers count
        dict(name="vb_small", kind="vb", n=1000, c=4.0, R=2, T=1.0, sweeps=256, spins=True),
        # the whole protocol on a fresh instance, once per disorder sample of a finite-size study:
        # create, attach, snapshots and log-spaced measurements to 2^10 sweeps, results, spins
        dict(name="vb_quench", kind="quench", n=4096, z=4, R=2, T=T_08_TC, sweeps=1024),
        # four replicas of a middling graph of odd size
        dict(name="vb_n20011_r4", kind="vb", n=20011, c=4.0, R=4, T=0.6, sweeps=128, spins=True),
        # the paper's own ensemble, random regular bipartite of degree 4, at the largest size of
        # the extrapolation chain
        dict(name="vb_rrbg", kind="vb", n=1 << 18, z=4, R=2, T=T_08_TC, sweeps=64),
        # one replica only (no overlap wanted), degree 3 on average, the configuration read back
        dict(name="vb_config_r1", kind="vb", n=300007, c=3.0, R=1, T=0.6, sweeps=32, spins=True),
        # window averages: every sweep is measured against every snapshot
        dict(name="vb_windows", kind="windows", n=1 << 20, c=4.0, R=2, T=1.0, sweeps=32),
        # the headline graph
        dict(name="vb_large", kind="vb", n=1 << 22, c=4.0, R=2, T=1.0, sweeps=64),
        # uneven graphs in lock-step, the configurations read back
        dict(name="vb_batch", kind="vb_batch", count=32, lo=10.0, hi=17.0, c=4.0, R=2, T=1.0,
             sweeps=128, spins=True),
        # the headline SK sample: 256 replicas sharing the couplings
        dict(name="sk_large", kind="sk", n=8192, R=256, T=0.4, block=128, sweeps=64),
        # a small SK sample of odd size with few replicas
        dict(name="sk_small", kind="sk", n=1001, R=32, T=0.6, block=128, sweeps=64, spins=True),
        # uneven SK samples in lock-step at two temperatures, block size left to the autotuner
        dict(name="sk_batch", kind="sk_batch", count=8, lo=9.0, hi=12.5, R=128, T=0.4, block=0,
             sweeps=32),
        # fields of given spins, all memory the caller's: a single call of a few tens of microseconds
        dict(name="sk_fields", kind="fields", n=2000, R=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng):
    kind = rng.choice(["vb"] * 5 + ["vb_batch", "windows", "quench"] + ["sk"] * 3 +
                      ["sk_batch", "fields"])
    T = rng.choice([0.6, 0.8, 1.0, T_08_TC])
    if kind == "vb":
        R = rng.choice([1, 2, 2, 2, 4])
        n = _log_int(rng, 1 << 10, (1 << 21) // max(1, R // 2))
        d = dict(kind=kind, n=n, R=R, T=T, sweeps=_log_int(rng, 16, 64),
                 spins=n < (1 << 19) and rng.random() < 0.5)
        if rng.random() < 0.25:
            d.update(n=n // 2 * 2, z=rng.choice([3, 4, 4]))  # bipartite: two equal halves
        else:
            d.update(c=rng.choice([3.0, 4.0, 4.0, 5.0]))
        return d
    if kind == "vb_batch":
        d = dict(kind=kind, R=rng.choice([1, 2, 2, 4]), T=T, sweeps=_log_int(rng, 16, 128))
        if rng.random() < 0.3:  # the graphs of one size of the bipartite ensemble, measured
            lo = math.log2(_log_int(rng, 1 << 13, 1 << 16) // 2 * 2)
            return dict(d, count=rng.randint(3, 16), lo=lo, hi=lo, z=4, spins=False)
        lo = rng.uniform(10.0, 12.0)
        return dict(d, count=rng.randint(3, 48), lo=lo, hi=lo + rng.uniform(1.0, 4.0), c=4.0, spins=True)
    if kind == "windows":
        return dict(kind=kind, n=_log_int(rng, 1 << 10, 1 << 20), c=4.0, R=rng.choice([2, 2, 4]), T=T,
                    sweeps=_log_int(rng, 16, 32))
    if kind == "quench":
        return dict(kind=kind, n=_log_int(rng, 1 << 10, 1 << 15) // 2 * 2, z=4, R=2, T=T,
                    sweeps=_log_int(rng, 256, 1024))
    if kind == "sk":
        return dict(kind=kind, n=_log_int(rng, 512, 8192), R=rng.choice([16, 32, 64, 128, 256]),
                    T=rng.choice([0.4, 0.6]), block=rng.choice([128, 128, 128, 0]),
                    sweeps=_log_int(rng, 16, 64), spins=rng.random() < 0.5)
    if kind == "sk_batch":
        lo = rng.uniform(9.0, 10.5)
        return dict(kind=kind, count=rng.randint(2, 8), lo=lo, hi=lo + rng.uniform(0.5, 2.0),
                    R=rng.choice([32, 64, 128]), T=rng.choice([0.4, 0.6]), block=rng.choice([0, 128]),
                    sweeps=_log_int(rng, 8, 32))
    return dict(kind="fields", n=_log_int(rng, 128, 2048), R=16 * rng.randint(1, 8))


# ------------------------------------------------------------------------------------ inputs
def _generator(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * seed + k)


def _csr(n, lo, hi, gen):
    """Symmetric CSR with one random 64-lane coupling word per undirected edge (host arrays)."""
    m = lo.numel()
    words = torch.randint(-(1 << 63), (1 << 63) - 1, (m,), generator=gen, device="cuda")
    src, dst = torch.cat([lo, hi]), torch.cat([hi, lo])
    order = torch.argsort(src * n + dst)  # the keys are distinct
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return dict(row_ptr=row_ptr.to(torch.int32).cpu().numpy(),
                col=dst[order].to(torch.int32).cpu().numpy(),
                jbits=torch.cat([words, words])[order].cpu().numpy().view(np.uint64))


def _poisson(n, c, gen):
    """A uniform simple graph with round(c n / 2) edges."""
    m = int(round(c * n / 2.0))
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        k = m - keys.numel() + 64 + (m - keys.numel()) // 32
        a = torch.randint(0, n, (k,), generator=gen, device="cuda")
        b = torch.randint(0, n, (k,), generator=gen, device="cuda")
        new = (torch.minimum(a, b) * n + torch.maximum(a, b))[a != b]
        keys = torch.unique(torch.cat([keys, new]))
    pick = torch.randperm(keys.numel(), generator=gen, device="cuda")[:m]
    keys = keys[pick]
    return _csr(n, keys // n, keys % n, gen)


def _regular(n, z, seed):
    """The paper's bipartite random regular graph."""
    row_ptr, col, eid = sg_inputs.random_regular_graph(n, z, seed, bipartite=True)
    return dict(row_ptr=row_ptr, col=col, jbits=sg_inputs.vb_lane_couplings(eid, n * z // 2, seed))


def _graph(case, n, seed, k=0):
    gen = _generator(seed, k)
    g = _regular(n, case["z"], 64 * seed + k) if "z" in case else _poisson(n, case["c"], gen)
    g.update(seed=1000003 * seed + k, temps=[case["T"]] * case["R"])
    return g


def _couplings(n, gen):
    b = torch.randint(0, 2, (n, n), generator=gen, device="cuda", dtype=torch.int8)
    upper = torch.triu(1 - 2 * b, diagonal=1)
    return upper + upper.T


def _sizes(case):
    """Sizes spread evenly over the logarithm of the case's range."""
    k = case["count"]
    return [int(round(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * (i + 0.5) / k)))
            for i in range(k)]


SNAPSHOTS = [0, 4, 16]  # waiting times of the stepped cases


def prepare(case, seed):
    kind, R = case["kind"], case["R"]
    if kind == "fields":
        gen = _generator(seed)
        J = _couplings(case["n"], gen)
        s = torch.randint(0, 2, (R, case["n"]), generator=gen, device="cuda", dtype=torch.int8) * 2 - 1
        h = torch.empty((R, case["n"]), dtype=torch.int32, device="cuda")
        return dict(case=case, J=J, s=s, h=h)
    if kind == "quench":
        tw, tm = sg_inputs.log_schedule([4, 16, 64], case["sweeps"])
        return dict(case=case, graph=_graph(case, case["n"], seed), tw=tw, tm=tm)
    if kind == "windows":
        run_ = sg.VBRun([_graph(case, case["n"], seed)], n_lanes=64, n_replicas=R, tw=[1, 2, 4, 8, 16],
                        windows=sg_inputs.geometric_windows(1, 1 << 20))
    elif kind == "vb":
        run_ = sg.VBRun([_graph(case, case["n"], seed)], n_lanes=64, n_replicas=R, tw=SNAPSHOTS)
    elif kind == "vb_batch":
        run_ = sg.VBRun([_graph(case, n, seed, k) for k, n in enumerate(_sizes(case))], n_lanes=64,
                        n_replicas=R, tw=SNAPSHOTS)
    elif kind == "sk":
        J = _couplings(case["n"], _generator(seed)).cpu().numpy()
        run_ = sg.SKRun(J, [case["T"]] * R, seed, block=case["block"], tw=SNAPSHOTS)
    else:
        samples = [dict(J=_couplings(n, _generator(seed, k)).cpu().numpy(), seed=1000003 * seed + k,
                        temps=[case["T"]] * (R // 2) + [1.5 * case["T"]] * (R // 2))
                   for k, n in enumerate(_sizes(case))]
        run_ = sg.SKBatchRun(samples, R, block=case["block"], tw=SNAPSHOTS)
    return dict(case=case, run=run_)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fields":
        sg.sg_sk_fields_noalloc(state["J"].data_ptr(), state["s"].data_ptr(), case["n"], case["R"],
                                state["h"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["h"]
    if kind == "quench":
        r = sg.VBRun([state["graph"]], n_lanes=64, n_replicas=case["R"], tw=state["tw"], tm=state["tm"])
        r.sweep(case["sweeps"])
        out = (*r.results(), r.spins()[0].view(np.int64))
        r.close()
        return out
    r = state["run"]
    r.sweep(case["sweeps"])
    if kind == "windows":
        return r.windows()
    if kind == "vb_batch" and case["spins"]:
        return [s.view(np.int64) for s in r.spins()]
    if case.get("spins"):
        s = r.spins()
        return (*r.measure(), s if kind == "sk" else s[0].view(np.int64))
    return r.measure()


def work(case):
    kind, R = case["kind"], case["R"]
    if kind == "fields":
        n = case["n"]
        return {"bytes": n * n + 5 * R * n, "flops": 2.0 * n * n * R}
    sweeps = case["sweeps"]
    if kind in ("sk", "sk_batch"):
        sizes = _sizes(case) if kind == "sk_batch" else [case["n"]]
        # per sweep: the couplings, one bit each, and the spins both ways; every flip moves all
        # fields, counted as the dense product of couplings and spin changes
        return {"bytes": sweeps * sum(n * n / 8 + 2 * R * n / 8 for n in sizes),
                "flops": sweeps * sum(2.0 * n * n * R for n in sizes)}
    n = sum(_sizes(case)) if kind == "vb_batch" else case["n"]
    degree = case.get("z") or case["c"]
    # per sweep: label and degree of every vertex, neighbour and coupling word of every directed
    # edge, spin words both ways; every snapshot of a measured sweep is read once
    per_sweep = 4 * n + 12 * degree * n + 16 * R * n
    if kind == "windows":
        per_sweep += 5 * 8 * R * n
    bytes_ = sweeps * per_sweep
    if case.get("spins"):
        bytes_ += 8 * R * n
    return {"bytes": bytes_, "flops": 0}


def exact(case, seed):
    """Spins and counts are integers that follow from the random numbers decision by decision:
    they have to be equal, and there is no value in 64 bits beside them.  The fields of given
    spins are a matrix product."""
    if case["kind"] != "fields":
        return None
    s = prepare(case, seed)
    return (s["s"].cpu().numpy().astype(np.int64) @ s["J"].cpu().numpy().astype(np.int64)).astype(np.int32)
