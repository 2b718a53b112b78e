"""Host models of what the CTA pairs' kernel adds to the stage protocol, and of tiles of different widths in sequence.

The pair: every CTA has its own loader, stage ring, two A-producer groups and epilogue; CTA 0's MMA warp issues for both and
its commits arrive in both CTAs, not necessarily at once.  The data barriers in CTA 0 are armed by both loaders and count
CTA 0's copies and CTA 1's half of B, so that CTA 0's producers, whose arrivals release, order the MMA after both halves;
CTA 1's data barriers count its row vectors only.  Barrier counts are the kernel's with one actor per warp group.  An
abort at any point leaves both loaders' copies to land: the exit path makes up for the arming of stages that only one of
them issued.

The widths: the accumulator's column halves are drained and overwritten separately, so the boundary between them has to
be the same for tiles of every width.  A boundary at half of each tile's own width is the negative control."""
import random

import pytest

from test_stage_protocol import Bar


def simulate_pair(NS, tiles, chunk, seed, full0_count=2, empty_count=2, b1_counted=True, abort_at=None):
    rng = random.Random(seed)
    ends = []                                  # per stage: does it end a drain chunk
    for nst in tiles:
        ends += [(k + 1) % chunk == 0 or k + 1 == nst for k in range(nst)]
    n, NF = len(ends), 2 * NS
    full = [[Bar(full0_count) for _ in range(NF)], [Bar(1) for _ in range(NF)]]
    empty = [[Bar(1) for _ in range(NS)] for _ in range(2)]
    a_full = [Bar(2), Bar(2)]
    acc_full, acc_empty = [Bar(1), Bar(1)], Bar(empty_count)
    landed = [dict(), dict(), dict()]          # buffer -> stage: CTA 0's copies, CTA 1's row vectors, CTA 1's half of B
    loaded, copies, arrivals = [0, 0], [], [[], []]
    prod = [[{"G": g, "data": True} for g in range(2)] for _ in range(2)]
    m = g_mma = completed = chunks = steps = 0  # completed: stages whose MMAs are done
    mma_queue, drained, g_epi = [], [0, 0], [0, 0]
    while not (drained[0] == drained[1] == sum(ends)):
        steps += 1
        assert steps < 400000, "no progress"
        if steps == abort_at:                  # every role stops here; the copies in flight land
            n0, n1 = loaded
            assert abs(n0 - n1) <= NS
            for k in range(min(n0, n1), max(n0, n1)):
                full[0][k % NF].arrive()
            for what, k in copies:
                full[what == 1][k % NF].complete_tx(1)
            for k in range(max(0, max(n0, n1) - NS), max(n0, n1)):
                assert full[0][k % NF].try_wait((k // NF) & 1), "exit path waits for copies that no barrier counts"
            return
        acts = []
        for c in range(2):
            k = loaded[c]
            if k < n and empty[c][k % NS].try_wait(((k // NS) & 1) ^ 1):
                acts.append(("load", c))
            for g, p in enumerate(prod[c]):
                G = p["G"]
                if G < n and (full[c][G % NF].try_wait((G // NF) & 1) if p["data"] else
                              G < 2 or empty[c][(G - 2) % NS].try_wait(((G - 2) // NS) & 1)):
                    acts.append(("prod", c, g))
            if arrivals[c]:
                acts.append(("arrive", c))
            if acc_full[c].try_wait(g_epi[c] & 1):
                acts.append(("epi", c))
        acts += [("land", i) for i in range(len(copies))]
        start = m < n and (m == 0 or ends[m - 1])
        if m < n and a_full[m & 1].try_wait((m >> 1) & 1) and (not start or acc_empty.try_wait((g_mma & 1) ^ 1)):
            acts.append(("issue",))
        if mma_queue:
            acts.append(("complete",))
        assert acts, f"deadlock at stage {m}"
        act = rng.choice(acts)
        if act[0] == "load":
            c, k = act[1], loaded[act[1]]
            assert completed >= k - NS + 1, "copy into a buffer the MMAs still read"
            for what in ((0,), (1, 2))[c]:
                landed[what].pop(k % NS, None)
                if what == 2 and not b1_counted:
                    copies.append((3, k))
                    continue
                full[what == 1][k % NF].arrive(tx=1)
                copies.append((what, k))
            loaded[c] += 1
        elif act[0] == "land":
            what, k = copies.pop(act[1])
            landed[min(what, 2)][k % NS] = k
            if what < 3:
                full[what == 1][k % NF].complete_tx(1)
        elif act[0] == "prod":
            c, p = act[1], prod[act[1]][act[2]]
            G = p["G"]
            if p["data"]:
                assert landed[c].get(G % NS) == G
                if c == 0:
                    assert landed[2].get(G % NS) == G, "CTA 0's producers do not order CTA 1's half of B"
            else:
                assert completed >= G - 1, "A slot stored while the MMAs read it"
                a_full[G & 1].arrive()
                p["G"] += 2
            p["data"] = not p["data"]
        elif act[0] == "issue":
            assert all(x.get(m % NS) == m for x in landed)
            if start:
                assert drained == [chunks, chunks], "accumulator overwritten before both CTAs drained it"
            mma_queue.append(m)
            if ends[m]:
                chunks += 1
                g_mma += 1
            m += 1
        elif act[0] == "complete":
            G = mma_queue.pop(0)
            completed = G + 1
            for c in range(2):
                arrivals[c] += ([("acc", G)] if ends[G] else []) + [("empty", G)]
        elif act[0] == "arrive":
            what, G = arrivals[act[1]].pop(0)
            (acc_full[act[1]] if what == "acc" else empty[act[1]][G % NS]).arrive()
        else:
            c = act[1]
            drained[c] += 1
            g_epi[c] += 1
            acc_empty.arrive()
    assert completed == n


def pair_tiles(rng):
    return [rng.randint(1, 20) for _ in range(4)]


@pytest.mark.parametrize("NS", [2, 3, 4, 5, 6])
def test_pair_protocol(NS):
    for seed in range(60):
        simulate_pair(NS, pair_tiles(random.Random(seed)), random.Random(seed).choice([1, 3, 16]), seed)


@pytest.mark.parametrize("NS", [2, 3, 4, 5, 6])
def test_pair_exit_after_an_abort(NS):
    for seed in range(200):
        rng = random.Random(seed)
        simulate_pair(NS, pair_tiles(rng), rng.choice([1, 3, 16]), seed, abort_at=rng.randint(1, 200))


@pytest.mark.parametrize("broken", [{"b1_counted": False, "full0_count": 1}, {"full0_count": 1}, {"empty_count": 1}])
def test_negative_controls_of_the_pair(broken):
    failures = 0
    for seed in range(60):
        try:
            simulate_pair(4, pair_tiles(random.Random(seed)), 3, seed, **broken)
        except AssertionError:
            failures += 1
    assert failures > 0


# ---------------------------------------------------------------------------
# Column halves of the accumulator: per tile (columns n, chunks), the MMAs write half h after acc_empty[h] and the
# epilogue drains it after acc_full[h]; blocks of 16 columns remember whose sums they hold.


def simulate_widths(tiles, boundary, seed):
    rng = random.Random(seed)
    acc_full, acc_empty = [Bar(1), Bar(1)], [Bar(1), Bar(1)]
    ops = []
    for t, (n, n_ch) in enumerate(tiles):
        lo = min(n, boundary(n))
        ops += [(h, (c0, c1), (t, ch)) for ch in range(n_ch) for h, (c0, c1) in enumerate(((0, lo), (lo, n))) if c1 > c0]
    held = [None] * 13                          # blocks of 16 of the 208 columns: undrained chunk
    g_mma, g_epi, commits = [0, 0], [0, 0], []
    i = e = 0
    for _ in range(100000):
        if e == len(ops):
            return
        acts = []
        if i < len(ops) and acc_empty[ops[i][0]].try_wait((g_mma[ops[i][0]] & 1) ^ 1):
            acts.append("mma")
        if commits:
            acts.append("commit")
        if acc_full[ops[e][0]].try_wait(g_epi[ops[e][0]] & 1):
            acts.append("epi")
        assert acts, "deadlock"
        a = rng.choice(acts)
        if a == "mma":
            h, (c0, c1), cid = ops[i]
            for b in range(c0 // 16, c1 // 16):
                assert held[b] is None, f"columns of {cid} still hold {held[b]}"
                held[b] = cid
            commits.append(h)
            g_mma[h] += 1
            i += 1
        elif a == "commit":
            acc_full[commits.pop(0)].arrive()
        else:
            h, (c0, c1), cid = ops[e]
            for b in range(c0 // 16, c1 // 16):
                assert held[b] == cid
                held[b] = None
            acc_empty[h].arrive()
            g_epi[h] += 1
            e += 1
    raise AssertionError("no progress")


def width_tiles(rng):
    return [(16 * rng.randint(1, 13), rng.randint(1, 3)) for _ in range(12)]


def test_one_boundary_of_the_column_halves_for_tiles_of_every_width():
    for seed in range(300):
        simulate_widths(width_tiles(random.Random(seed)), lambda n: 112, seed)


def test_negative_control_boundary_at_half_of_each_tile():
    failures = 0
    for seed in range(60):
        try:
            simulate_widths(width_tiles(random.Random(seed)), lambda n: (n // 2 + 15) // 16 * 16 if n >= 32 else n, seed)
        except AssertionError:
            failures += 1
    assert failures > 0
