"""The barrier protocol of the tensor-core expert GEMM that serves every batch of more than 64 tokens
(gemm_rows_kernel in csrc/gemm_rows.cu), modelled on the CPU. Two producers (one per CTA of the pair) walk a
ring whose stage count the launch chooses, over tiles of a contraction's k-blocks plus, where a segment has
adapters, some extra ones; both CTAs' bytes are counted on the leader's full[s]. The leader's MMA thread
consumes the stages in order, and its commits arrive on empty[s] and tfull[b] of both CTAs. Each CTA's eight
epilogue warps release an accumulator on the leader's tempty[b] (sixteen arrivals). At the end the leader's
producer waits for the stages still in flight, the peer's for their consumption, and then both CTAs may leave.

A wait passes when the barrier's phase has the other parity, as mbarrier.try_wait.parity does; every thread
keeps its stage and parity the way the kernel does (a stage counter that wraps and a parity bit that it
toggles). The model knows, besides, which phase each wait means: over random interleavings it checks that no
wait passes before that phase is complete, that nothing deadlocks, that every arrival and every landed copy
belongs to the phase under way, and that no copy is in flight and no stage unconsumed once the drains
return. Planted mistakes show that it can tell."""
import os
import random
import re

import pytest

from paper_2609_34077_gb300 import build

SRC = open(os.path.join(build.CSRC, "gemm_rows.cu")).read()


def _const(name, **known):
    expr = re.search(rf"constexpr int {name} = ([^;]+);", SRC).group(1)
    return int(eval(expr.replace("/", "//"), {}, known))  # noqa: S307 (integer constants of the source)


BK = _const("BK")
K_TILE_TOK = _const("kTileTok")
K_MAX_STAGES = _const("kMaxStages")
K_EPI_GROUPS = _const("kEpiGroups")
K_A_BYTES = _const("kABytes", BK=BK)
K_RING_BYTES = _const("kRingBytes", kABytes=K_A_BYTES, kTileTok=K_TILE_TOK, BK=BK)
EPI_WARPS = 4 * K_EPI_GROUPS  # of a CTA


def _stages(wide):
    """Stages of a launch whose widest token tile has `wide` tokens, as the kernel computes them."""
    stage = K_A_BYTES + wide // 2 * BK * 2
    n = min(K_MAX_STAGES, K_RING_BYTES // stage)
    assert n * stage <= K_RING_BYTES
    return n


class ProtocolError(AssertionError):
    pass


def _run(tiles, stages, seed, plant=None):
    """tiles: k-blocks of each of the pair's tiles. plant: a mistake in one of the threads."""
    rnd = random.Random(seed)
    total = sum(tiles)
    done = {}      # completed phases
    arrived = {}   # arrivals and landings of the phase under way
    flying = []    # copies under way: (rank, stage, round)
    commits = []   # commits in issue order (they complete in order): (kind, index, phase)
    arrivals = 8 if plant == "eight arrivals" else 2 * EPI_WARPS

    def passes(bar, parity, phase):
        """Whether a wait for `phase` (0-based; -1: nothing to wait for) of this parity passes now."""
        d = done.get(bar, 0)
        ok = (d & 1) != parity
        if ok and d < phase + 1:
            raise ProtocolError(f"wait on {bar} for phase {phase} passes with {d} complete")
        if not ok and d >= phase + 1:
            raise ProtocolError(f"wait on {bar} for phase {phase} missed it: {d} complete")
        return ok

    def arrive(bar, phase, what, need):
        d = done.get(bar, 0)
        if d != phase:
            raise ProtocolError(f"{what} of phase {phase} on {bar} during phase {d}")
        got = arrived.setdefault(bar, [])
        if what in got:
            raise ProtocolError(f"{what} twice in a phase of {bar}")
        got.append(what)
        if len(got) == need:
            arrived[bar] = []
            done[bar] = d + 1

    def producer(r):
        s = ph = issued = it = 0
        for nkb in tiles:
            for _ in range(nkb):
                while not passes(("empty", r, s), ph ^ 1, it // stages - 1):
                    yield False
                if r == 0:
                    arrive(("full", s), it // stages, "expect", 3)
                flying.append((r, s, it // stages))
                issued += issued < stages
                it += 1
                s += 1
                if s == stages:
                    s, ph = 0, ph ^ 1
                yield True
        for i in range(issued):  # oldest first
            back = issued - i
            j = s - back
            stage, parity = (j + stages, ph ^ 1) if j < 0 else (j, ph)
            if plant == "drain phase":
                parity = ph
            ring = ("full", stage) if r == 0 else ("empty", r, stage)
            while not passes(ring, parity, (it - back) // stages):
                yield False
            yield True
        if r == 0 and flying:
            raise ProtocolError("a copy is in flight after the leader's drain")
        if r == 1 and any(done.get(("empty", 1, x), 0) != (total - 1 - x) // stages + 1
                          for x in range(min(stages, total))):
            raise ProtocolError("a stage is unconsumed after the peer's drain")

    def mma():
        s = ph = it = 0
        for lt, nkb in enumerate(tiles):
            b = lt & 1
            while not passes(("tempty", b), ((lt >> 1) & 1) ^ 1, lt // 2 - 1):
                yield False
            if plant == "no extra blocks":  # the adapters' blocks forgotten on this side
                nkb = min(nkb, min(tiles))
            for _ in range(nkb):
                while not passes(("full", s), ph, it // stages):
                    yield False
                commits.append(("empty", s, it // stages))
                it += 1
                s += 1
                if s == stages:
                    s = 0
                    ph ^= plant != "parity kept"
                yield True
            commits.append(("tfull", b, lt // 2))

    def epilogue(r, warp):
        for lt in range(len(tiles)):
            b = lt & 1
            while not passes(("tfull", r, b), (lt >> 1) & 1, lt // 2):
                yield False
            arrive(("tempty", b), lt // 2, (r, warp), arrivals)
            yield True

    threads = {"p0": producer(0), "p1": producer(1), "mma": mma()}
    threads.update({f"e{r}{w}": epilogue(r, w) for r in (0, 1) for w in range(EPI_WARPS)})
    idle = set()
    while threads or flying or commits:
        names = [n for n in threads if n not in idle]
        choices = names + ["land"] * bool(flying) + ["commit"] * bool(commits)
        if not choices:
            raise ProtocolError("deadlock")
        n = rnd.choice(choices)
        if n == "land":
            r, s, rd = flying.pop(rnd.randrange(len(flying)))
            arrive(("full", s), rd, ("land", r), 3)
            idle.clear()
        elif n == "commit":
            kind, i, phase = commits.pop(0)
            for r in (0, 1):
                arrive((kind, r, i), phase, "commit", 1)
            idle.clear()
        else:
            try:
                if next(threads[n]):
                    idle.clear()
                else:
                    idle.add(n)
            except StopIteration:
                del threads[n]
                idle.clear()


# k-blocks of a pair's tiles: contraction, and contraction + the adapters' extra blocks
PATTERNS = [[1], [2] * 3, [11] * 4, [15, 21, 15, 15], [22, 24, 22], [3, 9, 9, 3, 3, 9], [64, 66], [1, 7] * 4]


@pytest.mark.parametrize("wide", [32, 64, 96, 128, 160, 192, 224, 256])
def test_random_interleavings(wide):
    for tiles in PATTERNS:
        for seed in range(6):
            _run(tiles, _stages(wide), seed)


def test_fewer_blocks_than_stages_and_exact_rounds():
    for stages in range(2, K_MAX_STAGES + 1):
        for n in range(1, 2 * stages + 2):
            _run([n], stages, n)
            _run([1] * n, stages, n)


@pytest.mark.parametrize("plant", ["eight arrivals", "drain phase", "no extra blocks", "parity kept"])
def test_planted_mistakes_are_found(plant):
    found = 0
    for seed in range(10):
        try:
            _run([15, 21, 15, 21], 7, seed, plant)
        except ProtocolError:
            found += 1
    assert found == 10


def test_the_kernel_has_the_modelled_counts():
    assert re.search(r"mbar_init\(&ctl->tempty\[b\], 8 \* kEpiGroups\)", SRC) and 2 * EPI_WARPS == 8 * K_EPI_GROUPS
    for bar in ("full", "empty"):
        assert re.search(rf"mbar_init\(&ctl->{bar}\[s\], 1\)", SRC)
    assert re.search(r"mbar_init\(&ctl->tfull\[b\], 1\)", SRC)
