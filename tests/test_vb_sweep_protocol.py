"""The grid-wide Viana-Bray sweep (csrc/vb_sweep.cu: k_vb_sweeps) on the CPU, at the level of its slices,
barriers and counters, over random interleavings of its warps.  A warp goes through (sweep, class, slice) with
one slice in work, the next one's words read ahead and the one after known; claimed slices are asked
for a slice before they are needed, and the counter moves at any time until the answer is used.  Checked:
every slice is updated once in every sweep, from its own words as the sweep before left them, while the
classes before it are done and the ones after it are not; a launch ends, also where a CTA's wait gives
up, and leaves its counters at zero.  Planted mistakes are caught: words of a warp's only slice not taken
over, the tail's first class not waited for, a CTA that arrives before its warps are done, one claim counter
for odd and even sweeps, groups of CTAs of which some have no CTA."""
import random
import re

import pytest


class ProtocolError(AssertionError):
    pass


class Cursor:
    def __init__(self, sweep, cls, slice_, had):
        self.sweep, self.cls, self.slice, self.had = sweep, cls, slice_, had

    def copy(self):
        return Cursor(self.sweep, self.cls, self.slice, self.had)


def launch(sizes, G, W, n_sweeps, claims, K, seed, mutant=None, give_up=None, max_steps=200000):
    rng = random.Random(seed)
    nc = len(sizes)
    cs = [sum(sizes[:c]) for c in range(nc + 1)]
    class_of = [c for c in range(nc) for _ in range(sizes[c])]
    version = [0] * cs[nc]
    stride = W * G
    tail = nc
    while tail > 0 and sizes[tail - 1] <= W:
        tail -= 1
    gbar, exits = [0], [0]
    counter = [[[0] * nc for _ in range(2)] for _ in range(K)]
    sync = [[0] * W for _ in range(G)]  # __syncthreads passed by each warp
    s_ok, stuck, waits = [True] * G, set(), [0] * G

    def classes_in_order(sweep, cls):
        for s, c in enumerate(class_of):
            want = sweep + 1 if c < cls else sweep
            if c != cls and version[s] != want:
                raise ProtocolError(f"class {cls} of sweep {sweep} beside class {c} at {version[s]}")

    def warp(b, w):
        gw, group = w * G + b, b % K
        group_warps = W * ((G - group + K - 1) // K)
        pending = [None]  # a claim asked for: its counter, and its number once that has moved

        def first(cls):
            return cs[cls] + (gw if cls < tail else w if b == 0 else W)

        def settle(c):
            while c.sweep < n_sweeps and c.slice >= cs[c.cls + 1]:
                c.cls += 1
                if c.cls == nc:
                    c.cls, c.sweep = 0, c.sweep + 1
                c.slice, c.had = first(c.cls), 0

        def claimed(c):
            return (claims and (G >= K or mutant == "empty_groups") and c.sweep < n_sweeps and c.had and c.cls < tail and
                    sizes[c.cls] > 2 * stride + K)

        def move():
            ctr, at = pending[0]
            pending[0] = (ctr, ctr[at])
            ctr[at] += 1

        def ask(c):
            if claimed(c):
                pending[0] = (counter[group][0 if mutant == "one_counter" else c.sweep & 1], c.cls)
                pending.append(True)  # not moved yet
                if rng.random() < 0.5:
                    move()
                    pending.pop()

        def claimed_slice(c):
            if len(pending) > 1:
                move()
                pending.pop()
            size = sizes[c.cls]
            a_sweep = (size - 2 * stride - group + K - 1) // K + group_warps
            v = pending[0][1] - (c.sweep if mutant == "one_counter" else c.sweep >> 1) * a_sweep
            if v < 0:
                raise ProtocolError("a claim counted in another sweep")
            return cs[c.cls] + 2 * stride + v * K + group if v < size else cs[c.cls + 1]

        def step(c):
            if claimed(c):
                c.slice = claimed_slice(c)
            else:
                c.slice += stride if c.cls < tail else W
                c.had = 1
            settle(c)
            ask(c)

        def own(c):
            return version[c.slice] if c.sweep < n_sweeps else None

        def syncthreads():
            sync[b][w] += 1
            n = sync[b][w]
            return lambda: min(sync[b]) >= n

        nx = Cursor(0, 0, first(0), 0)
        settle(nx)
        nn = nx.copy()
        step(nn)
        read_ahead = own(nx)
        yield None
        sweep = cls = phase = 0
        while sweep < n_sweeps:
            if phase > 0 and (cls < tail or cls == tail and mutant != "no_wait_at_tail") and G > 1:
                if w == 0:
                    waits[b] += 1
                    if give_up == (b, waits[b]):
                        s_ok[b] = False
                    else:
                        yield lambda: gbar[0] >= phase * G or b in stuck
                        s_ok[b] = gbar[0] >= phase * G
                yield syncthreads()
                if not s_ok[b]:
                    break
            while nx.sweep == sweep and nx.cls == cls:
                s, mine = nx.slice, read_ahead
                classes_in_order(sweep, cls)
                yield None  # the gathers are on their way
                nx = nn.copy()
                read_ahead = own(nx)
                yield None
                step(nn)
                yield None
                classes_in_order(sweep, cls)
                if mine != version[s] or mine != sweep:
                    raise ProtocolError(f"slice {s} updated from words of {mine}, it is at {version[s]} in sweep {sweep}")
                version[s] += 1
                if nx.slice == s and mutant != "no_forwarding":
                    read_ahead = version[s]
                yield None
            thin = tail <= cls and cls + 1 < nc
            if mutant == "early_arrival" and w == 0 and not thin:
                gbar[0] += 1
            yield syncthreads()
            if thin:
                cls += 1
                continue
            phase += 1
            if w == 0 and G > 1 and mutant != "early_arrival":
                gbar[0] += 1
            cls += 1
            if cls == nc:
                cls, sweep = 0, sweep + 1
        if w == 0:
            exits[0] += 1
            if exits[0] == G:
                gbar[0] = exits[0] = 0
                for g in counter:
                    for p in g:
                        p[:] = [0] * nc

    actors = {(b, w): warp(b, w) for b in range(G) for w in range(W)}
    waiting = dict.fromkeys(actors)
    for _ in range(max_steps):
        if not actors:
            break
        ready = [a for a in actors if waiting[a] is None or waiting[a]()]
        if not ready:
            if give_up is None or len(stuck) == G:
                raise ProtocolError("deadlock")
            stuck.add(rng.choice([b for b in range(G) if b not in stuck]))  # its wait runs out
            continue
        a = rng.choice(ready)
        try:
            waiting[a] = next(actors[a])
        except StopIteration:
            del actors[a]
    else:
        raise ProtocolError("step limit reached")
    if give_up is None and version != [n_sweeps] * cs[nc]:
        raise ProtocolError(f"slices updated {sorted(set(version))} times in {n_sweeps} sweeps")
    if gbar[0] or exits[0] or any(x for g in counter for p in g for x in p):
        raise ProtocolError("counters left behind")


# classes of a launch of 3 CTAs of 2 warps: several slices a warp, at most one, the tail on one CTA
SHAPES = [[30, 20, 5, 2, 1], [40], [17, 16], [27, 2, 2], [7, 1], [3, 3, 3], [19, 3, 18]]


@pytest.mark.parametrize("claims", [False, True])
@pytest.mark.parametrize("sizes", SHAPES)
def test_every_slice_once_a_sweep_in_class_order(sizes, claims):
    for seed in range(6):
        launch(sizes, 3, 2, 4, claims, 2, seed)
    launch(sizes, 1, 2, 3, claims, 2, 0)
    launch(sizes, 4, 1, 3, claims, 2, 1)


@pytest.mark.parametrize("claims", [False, True])
@pytest.mark.parametrize("give_up", [(0, 1), (1, 3), (2, 4)])
def test_a_wait_that_gives_up_ends_the_launch_and_rearms_it(claims, give_up):
    for seed in range(4):
        launch(SHAPES[0], 3, 2, 3, claims, 2, seed, give_up=give_up)


@pytest.mark.parametrize("mutant,sizes,match", [
    ("no_forwarding", [5], "updated from words of"),
    ("no_wait_at_tail", [30, 20, 2, 1], "beside class|updated from"),
    ("early_arrival", [30, 20, 2, 1], "beside class|updated from"),
    ("one_counter", [40], "another sweep|updated"),
    ("empty_groups", [40], "slices updated"),
])
def test_planted_mistakes_are_caught(mutant, sizes, match):
    caught = 0
    for seed in range(12):
        try:
            launch(sizes, 3, 2, 4, True, 5 if mutant == "empty_groups" else 2, seed, mutant=mutant)
        except ProtocolError as e:
            assert re.search(match, str(e)), str(e)
            caught += 1
    assert caught > 0
