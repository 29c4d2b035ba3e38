"""The warp that issues the matrix instructions of the fp32 table precompute (csrc/tables_mma.cu) and its neighbours, modelled on the
CPU: it takes two blocks at a time and gives both back behind the second one's products; the large products have an accumulator
on either side of the small ones', chunk by chunk in turn, and the small ones' lasts a tile.  Ring sizes and chunks are the source's."""
import os
import random
import re

from test_tables_ring_model import SOURCE, Barrier, ring_sizes


def chunk_size():
    with open(SOURCE) as f:
        return int(re.search(r"CHUNK = (\d+);", f.read()).group(1))


def run(stages, raw_stages, chunk, tiles, rng, wait_lo=True):
    """The first thing that goes wrong, or None.  tiles: their lengths in blocks."""
    full, empty = [[Barrier() for _ in range(stages)] for _ in range(2)]
    rfull, rempty = [[Barrier() for _ in range(raw_stages)] for _ in range(2)]
    accfull, accempty = [[Barrier() for _ in range(2)] for _ in range(2)]
    loempty = Barrier()
    raw, ring, flying, wrong = [None] * raw_stages, [None] * stages, [], []
    hi, lo, issued, sums = [[], []], [], [], []  # what the accumulators hold, commits still to take effect, the tiles' sums
    blocks = sum(tiles)

    def producer():
        for t in range(blocks):
            if t >= raw_stages:
                yield rempty[t % raw_stages], (t // raw_stages - 1) % 2
            flying.append(t)

    def half(h):
        for t in range(h, blocks, 2):
            s, r = t % stages, t % raw_stages
            yield rfull[r], t // raw_stages % 2
            got = raw[r]
            rempty[r].arrive()
            if t >= stages:
                yield empty[s], (t // stages - 1) % 2
            ring[s] = got
            full[s].arrive()

    def issuer():
        t = cc = 0
        for i, n in enumerate(tiles):
            if i > 0 and wait_lo:
                yield loempty, (i - 1) % 2
            for kb in range(0, n, chunk):
                slot = cc % 2
                if cc >= 2:
                    yield accempty[slot], (cc // 2 - 1) % 2
                end = t + min(chunk, n - kb)
                first = True
                while t < end:
                    pair = list(range(t, min(t + 2, end)))
                    for b in pair:
                        yield full[b % stages], b // stages % 2
                    for b in pair:
                        if ring[b % stages] != b:
                            wrong.append(f"block {ring[b % stages]} multiplied as block {b}")
                        hi[slot][:] = ([] if first else hi[slot]) + [b]
                        lo[:] = ([] if first and kb == 0 else lo) + [b]
                        first = False
                    issued.append([empty[b % stages] for b in pair])
                    t = end if len(pair) < 2 else t + 2
                issued.append([accfull[slot]])
                cc += 1

    def epilogue():
        cc = 0
        for n in tiles:
            large, small = [], []
            for kb in range(0, n, chunk):
                slot = cc % 2
                yield accfull[slot], cc // 2 % 2
                large += hi[slot]
                if kb + chunk >= n:
                    small += lo
                    loempty.arrive()
                accempty[slot].arrive()
                cc += 1
            sums.append((large, small))

    actors = {}
    for a in (producer(), half(0), half(1), issuer(), epilogue()):
        actors[a] = next(a, None)
    while not wrong:
        ready = [a for a, w in actors.items() if w is not None and w[0].passes(w[1])]
        steps = len(ready) + len(flying) + (1 if issued else 0)
        if steps == 0:
            break
        i = rng.randrange(steps)
        if i < len(ready):
            actors[ready[i]] = next(ready[i], None)
        elif i < len(ready) + len(flying):
            t = flying.pop(i - len(ready))
            raw[t % raw_stages] = t
            rfull[t % raw_stages].arrive()
        else:  # commits take effect in order
            for b in issued.pop(0):
                b.arrive()
    if wrong:
        return wrong[0]
    if any(w is not None for w in actors.values()):
        return "nothing moves any more"
    at = 0
    for n, (large, small) in zip(tiles, sums):
        if large != list(range(at, at + n)) or small != large:
            return f"a tile of {n} blocks: {large} and {small}"
        at += n
    return None


def faults(wait_lo=True):
    chunk, out = chunk_size(), []
    for seed in range(120):
        rng = random.Random(seed)
        tiles = [rng.choice([1, 2, 7, chunk, chunk + 1, 3 * chunk, 5 * chunk + 3])
                 for _ in range(rng.randint(1, 5))]
        out.append(run(*ring_sizes(), chunk, tiles, rng, wait_lo))
    return [f for f in out if f is not None]


def test_every_block_is_multiplied_once():
    assert faults() == []


def test_a_tile_that_does_not_wait_for_the_one_before_goes_wrong():
    assert faults(wait_lo=False) != []
