"""The streaming backward's teams, checked on the CPU: a model of one team
(its warps, the copies in flight, the stage barriers and the barrier at the
end of a group) under random interleavings. The warps take turns: the one whose
turn a group is (its number in the team's sequence modulo the warps) adds the
partial sums, refills the stage after a chunk's last group and updates the
slots; after a chance chunk warp 0 refills. No stage is refilled while a warp
still reads it, no partial sums are overwritten before their warp has added
them, no parity wait sees its barrier two phases ahead, and every warp
finishes. A warp that refills before the group's barrier, and partial sums in
one buffer, show the checker at work.
"""
import random

import pytest

STAGES = 2  # the kernel's kStreamStages


class Hazard(AssertionError):
    pass


def run(groups, warps, seed, refill_early=False, buffers=2):
    """groups[i]: groups of chunk i (0: a chance chunk, which has one barrier
    too). Returns once every warp has finished."""
    rng = random.Random(seed)
    full, sync, arrived = [0] * STAGES, [0], [0]  # phases completed; arrivals of the phase under way
    holds = [None] * STAGES                       # the chunk whose copies a stage takes or holds
    reading = [set() for _ in range(STAGES)]
    red = [None] * buffers                        # the group whose sums red[p] holds until their warp has read them
    copies = []                                   # stages with copies in flight

    def issue(i):
        s = i % STAGES
        if reading[s]:
            raise Hazard("stage refilled while read")
        holds[s] = i
        copies.append(s)

    def ready(done, k):
        if done >= k + 2:
            raise Hazard("barrier two phases ahead of a wait")
        return done >= k + 1

    def warp(w):
        phase = 0
        for i, n in enumerate(groups):
            s = i % STAGES
            while not ready(full[s], i // STAGES):
                yield
            assert holds[s] == i
            reading[s].add(w)
            for q in range(max(n, 1)):
                yield  # the members, from the stage
                last = q == max(n, 1) - 1
                turn = w == (phase % warps if n else 0)  # adds the sums, refills, updates
                if refill_early and last and turn and i + STAGES < len(groups):
                    issue(i + STAGES)
                if n:
                    if red[phase % buffers] not in (None, phase):
                        raise Hazard("partial sums overwritten")
                    red[phase % buffers] = phase
                if last:
                    reading[s].discard(w)
                if warps > 1:
                    arrived[0] += 1
                    if arrived[0] == warps:
                        arrived[0] = 0
                        sync[0] += 1
                    while not ready(sync[0], phase):
                        yield
                if turn:
                    if n:
                        yield  # the sums of the warps in order
                        if red[phase % buffers] != phase:
                            raise Hazard("partial sums of another group")
                        red[phase % buffers] = None
                    if last and i + STAGES < len(groups) and not refill_early:
                        issue(i + STAGES)
                    yield  # the update
                phase += 1

    for i in range(min(STAGES, len(groups))):
        issue(i)
    alive = [warp(w) for w in range(warps)]
    for _ in range(100000):
        if not alive:
            return
        k = rng.randrange(len(alive) + len(copies))
        if k < len(alive):
            try:
                next(alive[k])
            except StopIteration:
                alive.pop(k)
        else:
            full[copies.pop(k - len(alive))] += 1  # a chunk's copies land
    raise Hazard("a warp never finished")


@pytest.mark.parametrize("warps", [1, 2, 4, 8])
def test_no_interleaving_breaks_a_team(warps):
    for seed in range(150):
        rng = random.Random(1000 + seed)
        run([rng.choice([0, 1, 1, 2, 3]) for _ in range(rng.randint(1, 9))], warps, seed)


def test_a_refill_before_the_barrier_is_caught():
    with pytest.raises(Hazard):
        for seed in range(150):
            run([1, 2, 1, 2, 1, 2], 4, seed, refill_early=True)


def test_one_buffer_of_partial_sums_is_caught():
    # the next group's first warp can be there while this group's warp, another
    # one, has not read them yet
    with pytest.raises(Hazard):
        for seed in range(150):
            run([1, 2, 1, 2, 1, 2], 4, seed, buffers=1)


@pytest.mark.parametrize("groups", [[], [0], [1], [0] * 9, [3] * 9, [1, 0, 2, 0, 0, 3, 1]])
def test_sequences_at_the_edges(groups):
    for warps in (1, 3, 5, 8):
        for seed in range(30):
            run(groups, warps, seed)
