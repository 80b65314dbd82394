"""The waits of one chain CTA of the persistent SK sweep with the fields staged apart, on the CPU.

The staging warp fills a stage with the couplings and K* of block k as soon as the stage is released
and the spin-change ring has a free slot (`fullc`); the fields warp adds the fields of block k's rows
to the same stage once they are published (`fullh`).  A fold warp folds blocks k - L .. k - 3 when the
couplings are there, block k - 2 after its replica warp finished it (`cdone`), and needs the fields
only for the hand-over.  Model and checks as in test_sk_chain_protocol.py; in addition no stage's
fields are overwritten before the fold warps have read them, a fold warp folds only finished blocks in
either part, and a launch always finishes, also where the fields come late.  Planted mistakes (the
fields refilled without waiting for the stage, block k - 2 folded with the early part, the fields'
phase taken from the block's parity) are caught."""
import random
import re

import pytest

from test_sk_chain_protocol import MBar, ProtocolError

S, SLOTS = 3, 8


def run_cta(W, L, nk, seed, mutant=None, max_steps=400000):
    rng = random.Random(seed)
    fullc, fullh = [MBar(1) for _ in range(S)], [MBar(1) for _ in range(S)]
    emptyc = [MBar(2 * W) for _ in range(S)]
    cdone = [[MBar(1) for _ in range(2)] for _ in range(W)]
    hrdy = [[MBar(1) for _ in range(2)] for _ in range(W)]
    stage, fields = [None] * S, [None] * S
    users, readers = [set() for _ in range(S)], [set() for _ in range(S)]
    chain_done, done_cnt = [-1] * W, [0] * W
    applied, published, events = [0], [0], []

    def copy(k, dst, bar, who, inuse):
        s = k % S
        if inuse[s]:
            raise ProtocolError(f"stage {s} refilled for block {k} while in use")
        dst[s] = None
        inuse[s] = who
        bar[s].arrive_expect_tx(1)

        def land():
            dst[s] = k
            bar[s].complete_tx(1)
        events.append(land)

    def staging():
        for k in range(nk):
            if k >= S:
                yield lambda k=k: emptyc[k % S].done(k // S - 1)
            yield lambda k=k: applied[0] > k - SLOTS  # ring slot
            copy(k, stage, fullc, {("c", w) for w in range(W)} | {("f", w) for w in range(W)}, users)

    def fields_warp():
        for k in range(nk):
            if k >= S and mutant != "fields_without_release":
                yield lambda k=k: emptyc[k % S].done(k // S - 1)
            yield lambda k=k: k <= L or published[0] >= k - L
            copy(k, fields, fullh, set(range(W)), readers)

    def replica(w):
        for k in range(nk):
            s = k % S
            yield lambda k=k, s=s: fullc[s].done(k // S)
            yield lambda k=k: hrdy[w][k & 1].done(k >> 1)
            if stage[s] != k:
                raise ProtocolError(f"replica {w}: stage {s} holds {stage[s]}, expected {k}")
            chain_done[w], done_cnt[w] = k, k + 1
            cdone[w][k & 1].arrive()
            users[s].discard(("c", w))
            emptyc[s].arrive()

    def fold(w):
        def need(j, k):
            if j >= 0 and chain_done[w] < j:
                raise ProtocolError(f"fold {w}: block {j} folded for {k} before it was finished")
        for k in range(nk):
            s = k % S
            yield lambda k=k, s=s: fullc[s].done(k // S)
            if stage[s] != k:
                raise ProtocolError(f"fold {w}: stage {s} holds {stage[s]}, expected {k}")
            need(k - 2 if mutant == "early_part_too_long" else k - 3, k)
            if k >= 2:
                yield lambda k=k: cdone[w][k & 1].done((k - 2) >> 1)
            need(k - 2, k)
            ph = k & 1 if mutant == "fields_phase_from_parity" else k // S
            yield lambda s=s, ph=ph: fullh[s].done(ph)
            if fields[s] != k:
                raise ProtocolError(f"fold {w}: fields of {fields[s]}, expected {k}")
            readers[s].discard(w)
            hrdy[w][k & 1].arrive()
            users[s].discard(("f", w))
            emptyc[s].arrive()

    def field_ctas():
        for k in range(nk):
            yield lambda k=k: all(c > k for c in done_cnt)
            applied[0] = k + 1
            events.append(lambda k=k: published.__setitem__(0, max(published[0], k + 1)))

    actors = [staging(), fields_warp(), field_ctas()] + [f(w) for w in range(W) for f in (replica, fold)]
    live, waits = set(range(len(actors))), [None] * len(actors)
    for _ in range(max_steps):
        if not live and not events:
            return
        runnable = [i for i in live if waits[i] is None or waits[i]()]
        choices = runnable + (["event"] if events else [])
        if not choices:
            raise ProtocolError("deadlock: every warp waits and no copy is in flight")
        pick = rng.choice(choices)
        if pick == "event":
            events.pop(rng.randrange(len(events)))()
            continue
        try:
            waits[pick] = next(actors[pick])
        except StopIteration:
            live.discard(pick)
    raise ProtocolError("step limit reached")


@pytest.mark.parametrize("W", [1, 4, 8])
@pytest.mark.parametrize("L", [4, 6, 8])
def test_waits_are_consistent_and_finish(W, L):
    for seed in range(6):
        run_cta(W, L, nk=40, seed=seed)


@pytest.mark.parametrize("mutant,match", [
    ("fields_without_release", "refilled|fields of|ambiguous"),
    ("early_part_too_long", "folded for"),
    ("fields_phase_from_parity", "ambiguous|fields of|deadlock"),
])
def test_planted_mistakes_are_caught(mutant, match):
    caught = 0
    for seed in range(30):
        try:
            run_cta(4, 6, nk=40, seed=seed, mutant=mutant)
        except ProtocolError as e:
            assert re.search(match, str(e)), str(e)
            caught += 1
    assert caught > 0
