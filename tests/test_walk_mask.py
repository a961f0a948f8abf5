"""The shared masks of the on-demand walk (csrc/walk_mask.cuh) under schedules in which one CTA is late.

A model of the walk's scheme (csrc/walk_csc.cu; that of rounds in one launch is at the end): every CTA picks and decides a batch from
its own copy of the mask, tests its own candidates against the members kept, ORs the conflicts into a mask in global memory,
meets the others at a barrier and takes the mask over.  Word accesses of different CTAs are interleaved by a scheduler;
which words a batch writes and reads comes from the header itself, compiled for the host.  Whatever the schedule, every CTA
has to keep the first-fit list.  With one mask for all batches -- planted here, in the model -- a late reader does not."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WORD, BATCH = 4, 3                         # candidates per mask word and per batch (32 and 32 on the device)


@pytest.fixture(scope="module")
def mask_at(tmp_path_factory):
    d = tmp_path_factory.mktemp("walk_mask")
    src, lib = d / "m.cc", d / "m.so"
    src.write_text('#include "walk_mask.cuh"\nextern "C" int mask_at(unsigned int b, int pitch) { return strads::walk_mask_at(b, pitch); }\n'
                   'extern "C" int masks() { return strads::kWalkMasks; }\n'
                   'extern "C" int to_meet(unsigned int begun, unsigned int target) { return strads::walk_to_meet(begun, target); }\n')
    subprocess.run(["g++", "-x", "c++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1312_5766_b200", "csrc"),
                    "-o", str(lib), str(src)], check=True)
    so = ctypes.CDLL(str(lib))
    assert so.masks() == 2
    at = lambda batch, pitch: so.mask_at(ctypes.c_uint(batch), pitch)
    at.to_meet = lambda begun, target: bool(so.to_meet(ctypes.c_uint(begun), ctypes.c_uint(target)))
    return at


def _first_fit(conflict, n):
    kept = []
    for a in range(n):
        if not any(conflict[k][a] for k in kept):
            kept.append(a)
    return kept


def _cta(me, n_ctas, n, conflict, words, pitch, mask_at, arrived, kept):
    """One CTA as a generator: it yields before every access another CTA can see."""
    blocked = [False] * n
    cursor, batch = 0, 0
    while True:
        pick = [a for a in range(cursor, n) if not blocked[a]][:BATCH]
        if not pick:
            return
        new = []
        for a in pick:
            if not any(conflict[k][a] for k in new):
                new.append(a)
        kept += new
        cursor = pick[-1] + 1
        at = mask_at(batch, pitch)
        for b in range(me, n, n_ctas):     # the kept members against this CTA's own later candidates
            if not blocked[b] and any(k < b and conflict[k][b] for k in new):
                yield "run"
                words[at + b // WORD] |= 1 << (b % WORD)
        arrived[me] = batch + 1
        while min(arrived) < batch + 1:
            yield "wait"
        for w in range((n + WORD - 1) // WORD):
            yield "run"
            for i in range(WORD):
                if words[at + w] >> i & 1 and w * WORD + i < n:
                    blocked[w * WORD + i] = True
        batch += 1


def _walk(n, conflict, n_ctas, mask_at, order):
    """Runs the CTAs; `order` picks who takes the next step.  The kept list of every CTA, or None if a barrier gave up."""
    pitch = (n + WORD - 1) // WORD
    words = [0] * (2 * pitch)
    # (a CTA that has run out of batches arrives nowhere any more: whoever waits for it gives up, as on the device)
    arrived, kept = [0] * n_ctas, [[] for _ in range(n_ctas)]
    ctas = [_cta(i, n_ctas, n, conflict, words, pitch, mask_at, arrived, kept[i]) for i in range(n_ctas)]
    live, waited = set(range(n_ctas)), 0
    while live:
        i = order(sorted(live))
        state = next(ctas[i], "done")
        if state == "done":
            live.discard(i)
        waited = waited + 1 if state == "wait" else 0
        if waited > 1000:
            return None
    return kept


def _late(who, rng):
    """CTA `who` takes one step in twenty of its turns; the others run whenever they can."""
    return lambda live: who if who in live and (len(live) == 1 or rng.random() < 0.05) else rng.choice([i for i in live if i != who] or live)


def _cases():
    for seed in range(12):
        rng = random.Random(seed)
        n = rng.choice([5, 31, 32, 33, 64, 90])
        p = rng.choice([0.05, 0.2, 0.45])
        conflict = [[False] * n for _ in range(n)]
        for a in range(n):
            for b in range(a + 1, n):
                conflict[a][b] = conflict[b][a] = rng.random() < p
        yield seed, n, conflict


@pytest.mark.parametrize("n_ctas", [1, 2, 3, 5])
def test_every_cta_keeps_the_first_fit_list_whoever_is_late(mask_at, n_ctas):
    for seed, n, conflict in _cases():
        want = _first_fit(conflict, n)
        for who in range(n_ctas):
            got = _walk(n, conflict, n_ctas, mask_at, _late(who, random.Random(seed)))
            assert got is not None and all(k == want for k in got), (seed, n, who)


def test_one_mask_for_all_batches_would_not_do(mask_at):
    wrong = 0
    for seed, n, conflict in _cases():
        got = _walk(n, conflict, 3, lambda batch, pitch: 0, _late(1, random.Random(seed)))
        wrong += got is None or any(k != _first_fit(conflict, n) for k in got)
    assert wrong > 0


# Rounds in one launch (csrc/engine_csc.cuh): a CTA owns whole words of the mask and writes all of them after every batch, nothing is cleared
# (the masks hold whatever an earlier walk left), the next batch is picked from the mask alone, and the walk has no barrier before its
# first batch.  Around it what the walk must not overtake: the CTAs' shares of the last round's residual, which the products behind the walk
# read, and the word that says how a round is made, which CTA 0 changes when its walk is over.
def _rounds_cta(me, n_ctas, n, n_keep, conflict, n_rounds, mask_at, to_meet, g, out):
    pitch, target = (n + WORD - 1) // WORD, 0

    def meet():
        nonlocal target
        target += n_ctas
        yield "run"
        g["count"] += 1
        while not target <= g["count"] < target + n_ctas:
            yield "wait"

    for r in range(n_rounds):
        yield "run"
        g["applied"][me] = r
        yield "run"
        if g["avoid"] == 0:                # row buckets: two barriers, and a new count of rounds without them
            yield from meet()
            out["ways"][me].append("buckets")
            yield from meet()
            if me == 0:
                g["avoid"] = r % 3 + 1
        else:
            out["ways"][me].append("walk")
            begun, kept, cursor, batch, at = target, [], 0, 0, 0
            mine = {w: 0 for w in range(me, pitch, n_ctas)}
            while True:
                if batch == 0:
                    free = list(range(n))
                else:
                    blocked = []
                    for w in range(pitch):
                        yield "run"
                        blocked += [g["words"][at + w] >> i & 1 for i in range(WORD)]
                    free = [a for a in range(cursor, n) if not blocked[a]]
                if not free:
                    break
                new = []
                for a in free[:BATCH]:
                    if not any(conflict[k][a] for k in new):
                        new.append(a)
                new = new[:n_keep - len(kept)]
                kept += new
                cursor = free[:BATCH][-1] + 1
                if len(kept) == n_keep or len(free) <= BATCH:
                    break
                at = mask_at(batch, pitch)
                for w in mine:
                    for i in range(WORD):
                        b = w * WORD + i
                        mine[w] |= (b < n and b >= cursor and any(conflict[k][b] for k in new)) << i
                    yield "run"
                    g["words"][at + w] = mine[w]
                yield from meet()
                batch += 1
            if to_meet(begun, target):
                yield from meet()
            out["kept"][me].append(kept)
            yield "run"
            if me == 0:
                g["avoid"] -= 1
            out["late"] += any(a != r for a in g["applied"])          # (what the products would read)
        yield from meet()
        yield from meet()


def _rounds(n, n_keep, conflict, n_ctas, mask_at, to_meet, who, seed):
    rng = random.Random(seed)
    g = dict(count=0, avoid=2, applied=[-1] * n_ctas, words=[rng.randrange(1 << WORD) for _ in range(2 * ((n + WORD - 1) // WORD))])
    out = dict(ways=[[] for _ in range(n_ctas)], kept=[[] for _ in range(n_ctas)], late=0)
    ctas = [_rounds_cta(i, n_ctas, n, n_keep, conflict, 6, mask_at, to_meet, g, out) for i in range(n_ctas)]
    order, live, waited = _late(who, rng), set(range(n_ctas)), 0
    while live:
        i = order(sorted(live))
        state = next(ctas[i], "done")
        if state == "done":
            live.discard(i)
        waited = waited + 1 if state == "wait" else 0
        if waited > 1000:
            return False
    want = _first_fit(conflict, n)[:n_keep]
    return out["late"] == 0 and all(w == out["ways"][0] for w in out["ways"]) and all(k == want for ks in out["kept"] for k in ks)


@pytest.mark.parametrize("n_ctas", [1, 2, 3, 5])
def test_rounds_in_one_launch_whoever_is_late(mask_at, n_ctas):
    for seed, n, conflict in _cases():
        for n_keep in (1, BATCH, 8, n):        # walks that end with their first batch, without a barrier, and that do not
            for who in range(n_ctas):
                assert _rounds(n, n_keep, conflict, n_ctas, mask_at, mask_at.to_meet, who, seed), (seed, n, n_keep, who)


def test_walks_without_a_barrier_would_not_do(mask_at):
    assert not all(_rounds(n, 1, conflict, 3, mask_at, lambda begun, target: False, who, seed) for seed, n, conflict in _cases() for who in range(3))
    assert not all(_rounds(n, 8, conflict, 3, lambda batch, pitch: 0, mask_at.to_meet, who, seed) for seed, n, conflict in _cases() for who in range(3))
