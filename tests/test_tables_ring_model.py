"""The shared-memory rings of the fp32 table precompute (csrc/tables_mma.cu), modelled on the CPU: copies that land in any
order, two halves of converting warps that take blocks in turn, products in order, and barriers that are waited for by the
parity of a phase alone.  The ring sizes are the source's."""
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_20375_b200", "csrc",
                      "tables_mma.cu")


class Barrier:
    """Phases completed so far; one arrival completes a phase."""

    def __init__(self):
        self.done = 0

    def arrive(self):
        self.done += 1

    def passes(self, parity):  # mbarrier.try_wait.parity: the phase that is not complete yet has the other parity
        return self.done % 2 != parity


def run(stages, raw_stages, blocks, rng, late):
    """The first thing that goes wrong, or None.  late: the block whose copy lands when nothing else can move, or None."""
    full, empty = [[Barrier() for _ in range(stages)] for _ in range(2)]
    rfull, rempty = [[Barrier() for _ in range(raw_stages)] for _ in range(2)]
    raw, ring, flying, wrong = [None] * raw_stages, [None] * stages, [], []

    def producer():
        for t in range(blocks):
            s = t % raw_stages
            if t >= raw_stages:
                yield rempty[s], (t // raw_stages - 1) % 2
            flying.append(t)

    def half(h):
        for t in range(h, blocks, 2):
            s, r = t % stages, t % raw_stages
            yield rfull[r], t // raw_stages % 2
            got = raw[r]
            if got != t:
                wrong.append(f"block {got} converted as block {t}")
            rempty[r].arrive()
            if t >= stages:
                yield empty[s], (t // stages - 1) % 2
            ring[s] = got
            full[s].arrive()

    def products():
        for t in range(blocks):
            s = t % stages
            yield full[s], t // stages % 2
            if ring[s] != t:
                wrong.append(f"block {ring[s]} multiplied as block {t}")
            empty[s].arrive()

    actors = {}
    for a in (producer(), half(0), half(1), products()):
        actors[a] = next(a, None)
    while True:
        ready = [a for a, w in actors.items() if w is not None and w[0].passes(w[1])]
        landing = [t for t in flying if t != late]
        if not ready and not landing:
            landing = list(flying)
        if wrong or not (ready or landing):
            break
        i = rng.randrange(len(ready) + len(landing))
        if i < len(ready):
            actors[ready[i]] = next(ready[i], None)
        else:
            t = landing[i - len(ready)]
            flying.remove(t)
            raw[t % raw_stages] = t
            rfull[t % raw_stages].arrive()
    if wrong:
        return wrong[0]
    return "nothing moves any more" if any(w is not None for w in actors.values()) else None


def faults(stages, raw_stages):
    out = []
    for seed in range(300):
        rng = random.Random(seed)
        out.append(run(stages, raw_stages, 60, rng, rng.randrange(60) if seed % 3 else None))
    return [f for f in out if f is not None]


def ring_sizes():
    with open(SOURCE) as f:
        m = re.search(r"STAGES = (\d+), RAW_STAGES = F32 \? (\d+) : 1;", f.read())
    return int(m.group(1)), int(m.group(2))


def test_no_copy_is_too_late_for_the_rings():
    assert faults(*ring_sizes()) == []


@pytest.mark.parametrize("stages,raw_stages", [(4, 5), (4, 3)])
def test_rings_of_odd_size_go_wrong(stages, raw_stages):
    """... so the model sees what it is there for: a half that waits on every second phase takes a stage for full while its copy
    is on the way."""
    assert faults(stages, raw_stages) != []
