"""The barriers of the flow decoder's cluster step (csrc/dc_cluster_sync.h, compiled for the host): however late loads and signals land and however warps and
CTAs are interleaved, no warp passes a wait for a K/V block that has not landed, and no CTA reads a row before the signal of the CTA that wrote it."""
import ctypes
import os
import random
import subprocess

import pytest

import paper_2609_35115_b200 as dc

SRC = """
#include "dc_cluster_sync.h"
extern "C" {
unsigned kv_slots() { return dc::CLU_KVS; }
int kv_item(int i, int n) { bool v; int b; dc::clu_item(i, n, &v, &b); return 2 * b + v; }
int kv_item_k(int b) { return dc::clu_item_k(b); }
int kv_item_v(int b, int n) { return dc::clu_item_v(b, n); }
unsigned kv_full(int is_v, unsigned slot) { return dc::clu_kv_full(is_v != 0, slot); }
unsigned hand(unsigned n) { return dc::clu_hand(n); }
unsigned hand_parity(unsigned n) { return dc::clu_hand_parity(n); }
unsigned kv_next(unsigned* bits, unsigned slot) { dc::CluKvPhases p; p.bits = *bits; const unsigned r = p.next(slot); *bits = p.bits; return r; }
}
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("cluster_sync")
    (d / "ring.cpp").write_text(SRC)
    csrc = os.path.join(os.path.dirname(dc.__file__), "csrc")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", csrc, "-o", str(d / "ring.so"), str(d / "ring.cpp")], check=True)
    return ctypes.CDLL(str(d / "ring.so"))


class Early(Exception):
    pass


def walk(ring, jobs, rng, shared=False):
    """One interleaving of the loader, the scores' warp, the softmax and the output's warp over jobs of so many key blocks each.  A barrier is the number of
    its completed phases; a wait with parity p passes while that number's parity differs.  `shared`: one full barrier per slot, waited for by item number."""
    slots = ring.kv_slots()
    full, empty = [0] * (2 * slots), [0] * slots
    content, pending = [None] * slots, []            # landed item of a slot; (slot, barrier, item) under way
    blocks = [(j, b) for j, n in enumerate(jobs) for b in range(n)]
    first = [2 * sum(jobs[:j]) for j in range(len(jobs))]
    items = [(j, i) for j, n in enumerate(jobs) for i in range(2 * n)]
    order = {}
    for j, i in items:
        k = ring.kv_item(i, jobs[j])
        order[first[j] + i] = (j, k >> 1, k & 1)
    for j, b in blocks:                              # the three functions describe one order
        assert order[first[j] + ring.kv_item_k(b)] == (j, b, 0) and order[first[j] + ring.kv_item_v(b, jobs[j])] == (j, b, 1)

    at = dict(load=0, k=0, soft=0, v=0)
    bits = dict(k=ctypes.c_uint(0), v=ctypes.c_uint(0))
    next_parity = {}                                 # of a warp that polls: taken once per wait

    def passes(count, parity):
        return (count & 1) != parity

    def load():
        j, i = items[at["load"]]
        gi = first[j] + i
        slot, k = gi % slots, gi // slots
        if k > 0 and not passes(empty[slot], (k - 1) & 1):
            return False
        content[slot] = None
        pending.append((slot, slot if shared else ring.kv_full(order[gi][2], slot), gi))
        at["load"] += 1
        return True

    def consume(who, is_v):
        j, b = blocks[at[who]]
        if is_v and at["soft"] <= at["v"]:           # P(b) has to be there
            return False
        if not is_v and at["k"] - at["soft"] >= 2:   # the stream's previous scores have been read
            return False
        gi = first[j] + (ring.kv_item_v(b, jobs[j]) if is_v else ring.kv_item_k(b))
        slot = gi % slots
        if who not in next_parity:
            next_parity[who] = (gi // slots) & 1 if shared else ring.kv_next(ctypes.byref(bits[who]), slot)
        if who not in passed and not passes(full[slot if shared else ring.kv_full(is_v, slot)], next_parity[who]):
            return False
        if content[slot] != gi:
            raise Early((jobs, j, b, "V" if is_v else "K"))
        next_parity.pop(who)
        passed.discard(who)
        empty[slot] += 1
        at[who] += 1
        return True

    def poll_v():                                    # the output's warp polls for its V block before it waits for P
        if at["v"] < len(blocks) and "v" not in passed:
            j, b = blocks[at["v"]]
            gi = first[j] + ring.kv_item_v(b, jobs[j])
            slot = gi % slots
            if "v" not in next_parity:
                next_parity["v"] = (gi // slots) & 1 if shared else ring.kv_next(ctypes.byref(bits["v"]), slot)
            if passes(full[slot if shared else ring.kv_full(True, slot)], next_parity["v"]):
                passed.add("v")

    passed = set()
    while at["v"] < len(blocks):
        poll_v()
        moves = []
        if at["load"] < len(items):
            moves.append("load")
        if at["k"] < len(blocks):
            moves.append("k")
        if at["soft"] < at["k"] and at["soft"] - at["v"] < 2:
            moves.append("soft")
        moves.append("v")
        rng.shuffle(moves)
        if pending and rng.random() < 0.3:
            moves.insert(0, "land")
        elif pending:
            moves.append("land")
        for m in moves:
            if m == "load":
                done = load()
            elif m == "land":
                slot, bar, gi = pending.pop(rng.randrange(len(pending)))
                content[slot] = gi
                full[bar] += 1
                done = True
            elif m == "soft":
                at["soft"] += 1
                done = True
            else:
                done = consume(m, m == "v")
            if done:
                break
        else:
            raise AssertionError("no move is left")


JOBS = [[n] for n in range(1, 12)] + [[5, 5, 5], [4, 1, 6], [1, 1, 1, 1], [2, 3, 2, 5], [6, 6]]


@pytest.mark.parametrize("jobs", JOBS, ids=str)
def test_no_wait_passes_before_its_block_has_landed(ring, jobs):
    for seed in range(300):
        walk(ring, jobs, random.Random(seed))


def test_the_walk_finds_one_barrier_for_both_kinds(ring):
    """The same walk over one full barrier per slot, whose phases two warps share: from four key blocks on it finds the V block that is multiplied early."""
    def early(jobs):
        for seed in range(300):
            try:
                walk(ring, jobs, random.Random(seed), shared=True)
            except Early:
                return True
        return False

    assert [early([n]) for n in range(1, 7)] == [False, False, False, True, True, True]
    assert early([5, 5])


def walk_hand(ring, stages, ctas, rng, form="two"):
    """One interleaving of the loaders' and the epilogues' warps of a cluster over stages that hand over in bulk ("b"), in bulk with row statistics for the next
    stage ("s"), or behind a fence ("f").  A row is visible to a CTA from the writer's signal on; "two": as in the kernel, "one": a single barrier,
    "none": only the cluster barrier between a stage and the next."""
    nth, n = [], 0                                   # of a stage: how many in bulk came before it
    for kind in stages:
        nth.append(n)
        n += kind != "f"
    index = (lambda j: 0) if form == "one" else ring.hand
    parity = (lambda j: j & 1) if form == "one" else ring.hand_parity
    phase = [[0, 0] for _ in range(ctas)]            # completed phases of a CTA's barriers
    armed, tx = [[False, False] for _ in range(ctas)], [[0, 0] for _ in range(ctas)]
    seen = [set() for _ in range(ctas)]              # (stage, writer) of the signals that have landed
    flying = []
    arrived = [0] * len(stages)                      # at the cluster barrier behind a stage; two warps of every CTA

    def settle(c, i):
        if armed[c][i] and tx[c][i] == 0:
            phase[c][i] += 1
            armed[c][i] = False

    def passes(c, j):
        return (phase[c][index(j)] & 1) != parity(j)

    def check(c, k):
        if any((k, w) not in seen[c] for w in range(ctas)):
            raise Early((c, k))

    requested = [0] * ctas                           # operands: of the stages before this number

    def loader(c):
        requested[c] = 1
        for k, kind in enumerate(stages):
            if kind != "f" and form != "none":
                i = index(nth[k])
                assert not armed[c][i], "the phase before is still open"
                tx[c][i] += ctas
                armed[c][i] = True
                settle(c, i)
            arrived[k] += 1
            yield lambda: True
            if kind != "f" and form != "none":
                yield lambda: passes(c, nth[k])
            else:
                yield lambda: arrived[k] == 2 * ctas
            if kind != "f":
                check(c, k)
            requested[c] = k + 2
            yield lambda: arrived[k] == 2 * ctas

    def epilogue(c):
        for k, kind in enumerate(stages):
            yield lambda: requested[c] > k
            if k > 0 and stages[k - 1] == "s":
                if form != "none":
                    yield lambda: passes(c, nth[k - 1])
                check(c, k - 1)
            yield lambda: True                       # the products
            if kind != "f":
                flying.extend((k, c, d) for d in range(ctas))
            arrived[k] += 1
            yield lambda: arrived[k] == 2 * ctas

    warps = [w(c) for c in range(ctas) for w in (loader, epilogue)]
    ready = [next(w) for w in warps]
    slow = rng.choice([0.02, 0.2, 0.6])
    while warps:
        can = [i for i, r in enumerate(ready) if r()]
        if flying and (not can or rng.random() < slow):
            k, c, d = flying.pop(rng.randrange(len(flying)))
            seen[d].add((k, c))
            if form != "none":
                i = index(nth[k])
                tx[d][i] -= 1
                settle(d, i)
            continue
        assert can, "no move is left"
        i = rng.choice(can)
        try:
            ready[i] = next(warps[i])
        except StopIteration:
            del warps[i], ready[i]


# input, conv blocks, projections, attention (in bulk or behind a fence), output projection, output
HAND_STAGES = {"one job": "bbsfbbbsfbsf" * 3, "several jobs": "bbsffbbsffsf" * 3, "short": "bsfbsf" * 4}


@pytest.mark.parametrize("stages", HAND_STAGES.values(), ids=HAND_STAGES.keys())
@pytest.mark.parametrize("ctas", [2, 5])
def test_no_row_is_read_before_its_writers_signal(ring, stages, ctas):
    for seed in range(60):
        walk_hand(ring, stages, ctas, random.Random(seed))


@pytest.mark.parametrize("form", ["none", "one"])
def test_the_walk_finds_the_cluster_barrier_alone_and_a_single_barrier(ring, form):
    found = 0
    for seed in range(60):
        try:
            walk_hand(ring, HAND_STAGES["one job"], 4, random.Random(seed), form)
        except (Early, AssertionError):
            found += 1
    assert found > 0
