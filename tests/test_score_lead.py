"""Liveness of the two-pass score kernel's chunk schedule and the bound on its chunk records, on the CPU.

Chunks are dealt round-robin to the CTAs.  In a CTA, pass 1 takes its chunks in order and may be at
most `lead` tile slots ahead of pass 2; pass 2 of a chunk waits until pass 1 and the value norms of
its whole head (in split mode of both halves) are published.  The conditions only ever become true,
so "some CTA can always move until all are done" does not depend on timing.  A chunk record lives in a
ring of 16: pass 1 may never be more than 13 chunks ahead of pass 2.
"""
import random

import pytest

TILE, RING, MAX_LEAD_CHUNKS = 128, 16, 12


def ceil_div(a, b):
    return -(-a // b)


def run(seq, layers, heads, split, window, radius, chunk_tiles, grid, extra, lead=None):
    units, out_keys = heads << split, TILE - 2 * radius
    cph = [ceil_div(ceil_div(n, TILE), chunk_tiles) for n in seq]
    slots = ceil_div(chunk_tiles * TILE, out_keys) + 2
    longest = max(cph) << split
    if lead is None:
        need = slots * ((longest - 1) // grid) + chunk_tiles
        lead = min(need + extra, MAX_LEAD_CHUNKS * slots)
    chunks = []                                      # (value-norm head, its chunks, pass-1, pass-2 tiles)
    for layer in range(layers):
        for b, n in enumerate(seq):
            for u in range(units):
                for i in range(cph[b]):
                    share = lambda t: t // cph[b] + (1 if i < t % cph[b] else 0)
                    n1, n2 = share(ceil_div(n, TILE)), share(ceil_div(max(n - window, 0), out_keys))
                    assert n1 <= chunk_tiles and n2 <= slots
                    chunks.append(((layer, b, u >> split), cph[b] << split, n1, n2))
    mine = [chunks[c::grid] for c in range(grid)]
    p1, p2 = [[0, 0] for _ in range(grid)], [[0, 0] for _ in range(grid)]   # (chunk, tile)
    published, moved = {}, True
    while moved:
        moved = False
        for c in range(grid):
            while p1[c][0] < len(mine[c]):
                j, t = p1[c]
                at2 = p2[c][0] * slots + p2[c][1] if p2[c][0] < len(mine[c]) else 1 << 40
                if j * slots + t > at2 + lead:
                    break
                assert j - p2[c][0] <= MAX_LEAD_CHUNKS + 1 < RING - 2
                p1[c][1] += 1
                if p1[c][1] == mine[c][j][2]:
                    published[mine[c][j][0]] = published.get(mine[c][j][0], 0) + 1
                    p1[c] = [j + 1, 0]
                moved = True
            if p2[c][0] < len(mine[c]):
                j, t = p2[c]
                head, want, _, n2 = mine[c][j]
                if published.get(head, 0) == want:
                    p2[c] = [j, t + 1] if t + 1 < n2 else [j + 1, 0]
                    moved = True
    return all(p1[c][0] == p2[c][0] == len(mine[c]) for c in range(grid))


@pytest.mark.parametrize("seed", range(40))
def test_every_wait_ends(seed):
    rng = random.Random(seed)
    seq = [rng.randint(16, 60 * TILE) for _ in range(rng.randint(1, 5))]
    if rng.random() < 0.3:
        seq[rng.randrange(len(seq))] = 16            # window only: nothing to score
    assert run(seq, layers=rng.randint(1, 3), heads=rng.choice([1, 2, 4]), split=rng.randint(0, 1),
               window=16, radius=rng.choice([0, 2, 3, 31]), chunk_tiles=rng.randint(4, 16),
               grid=rng.randint(4, 24), extra=rng.choice([0, 8, 12]))


def test_too_short_a_lead_is_caught():
    assert not run([6000], 1, 2, 0, 16, 3, chunk_tiles=4, grid=3, extra=0, lead=2)
