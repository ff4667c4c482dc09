"""A model of the barriers that join the roles of the many-token projection
(gemm_tc.cu), with the rings that the library reports for every token tile and
group size: whichever role is slow, held back once anywhere or behind at every
step, all roles come to their end, and no wait by parity lets a role through
before the phase it means.  A ring whose barriers another role can pass by two
phases would stand here (a parity wait tells neighbouring phases only).
No GPU."""
import os

import pytest

import paper_2608_19147_gb300 as pkg
from paper_2608_19147_gb300 import build as libbuild

EPI_WARPS, DQ_WARPS = 8, 4  # epilogue warps; warps per dequantise set


@pytest.fixture(scope="module", autouse=True)
def _library():
    try:
        libbuild.build()
    except RuntimeError as e:  # no nvcc here
        if not os.path.exists(libbuild.LIB):
            pytest.skip(str(e))
    pkg.load_library()


class Bar:
    """An mbarrier: `phase` completed phases; a phase ends when all arrivals have come (a copy's bytes count as one)."""

    def __init__(self, count):
        self.count = self.left = count
        self.phase = 0

    def arrive(self):
        self.left -= 1
        assert self.left >= 0
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1


class Model:
    """The roles as generators: a yielded (barrier, phase) is a wait for that phase, None an operation's end."""

    def __init__(self, steps, G, rings):
        self.steps, self.G = steps, G
        self.US, self.BS, self.AS, self.D, self.mma_warps, self.dq_sets = rings
        self.u_full = [Bar(2) for _ in range(self.US)]  # the producer's arrival and the bytes
        self.u_empty = [Bar(DQ_WARPS + EPI_WARPS) for _ in range(self.US)]
        self.full = [Bar(DQ_WARPS + 2) for _ in range(self.BS)]
        self.done = [Bar(1) for _ in range(self.BS * G)]
        self.d_empty = [Bar(EPI_WARPS) for _ in range(self.D)]
        self.copies, self.pipe = [], []  # barriers to arrive on: copies in flight, the tensor pipe's commits in order
        self.actors = {"producer": self.producer()}
        self.actors.update({"mma%d" % w: self.mma(w) for w in range(self.mma_warps)})
        self.actors.update({"dq%d.%d" % (s, w): self.dq(s) for s in range(self.dq_sets) for w in range(DQ_WARPS)})
        self.actors.update({"epi%d" % w: self.epi() for w in range(EPI_WARPS)})
        self.actors.update({"copy": self.engine(self.copies), "pipe": self.engine(self.pipe)})
        self.at = {a: next(g, "end") for a, g in self.actors.items()}

    def wait_done(self, k, gq):
        return self.done[k % self.BS * self.G + gq], k // self.BS

    def producer(self):
        def units(k):
            self.u_full[k % self.US].arrive()
            self.copies.append(self.u_full[k % self.US])

        for k in range(min(self.US, self.steps)):
            units(k)
        for k in range(self.steps):
            if k >= self.US:
                yield self.u_empty[k % self.US], k // self.US - 1
                units(k)
            if k >= self.BS:
                yield self.wait_done(k - self.BS, self.G - 1)
            self.full[k % self.BS].arrive()
            self.copies.append(self.full[k % self.BS])
            yield None

    def mma(self, w):
        for k in range(w, self.steps, self.mma_warps):
            yield self.full[k % self.BS], k // self.BS
            for gq in range(self.G):
                q = k * self.G + gq
                if q >= self.D:
                    yield self.d_empty[q % self.D], q // self.D - 1
                self.pipe.append(self.done[k % self.BS * self.G + gq])
                yield None

    def dq(self, s):
        for k in range(s, self.steps, self.dq_sets):
            yield self.u_full[k % self.US], k // self.US
            if k >= self.AS:
                yield self.wait_done(k - self.AS, self.G - 1)
            self.u_empty[k % self.US].arrive()
            self.full[k % self.BS].arrive()
            yield None

    def epi(self):
        for k in range(self.steps):
            yield self.u_full[k % self.US], k // self.US
            self.u_empty[k % self.US].arrive()  # the step's scales are in registers
            for gq in range(self.G):
                yield self.wait_done(k, gq)
                self.d_empty[(k * self.G + gq) % self.D].arrive()
                yield None

    @staticmethod
    def engine(queue):
        while True:
            yield queue  # runs while the queue holds something
            queue.pop(0).arrive()

    def step(self, name):
        """One operation of a role, if it can go on."""
        at = self.at[name]
        if at == "end":
            return False
        if isinstance(at, tuple):
            bar, phase = at
            if bar.phase % 2 == phase % 2:  # by parity
                return False
            assert bar.phase > phase, "%s passed a wait early" % name
        elif isinstance(at, list) and not at:
            return False
        self.at[name] = next(self.actors[name], "end")
        return True

    def settle(self, names):
        """All of `names` as far as they go."""
        went, any_ = True, False
        while went:
            went = False
            for n in names:
                while self.step(n):
                    went = any_ = True
        return any_

    def finish(self, slow, after):
        """`slow` acts only when nobody else can (from its operation `after` on, for one operation or for good)."""
        rest = [n for n in self.actors if n not in slow]
        n = 0
        while True:
            if after is None or n == after:
                self.settle(rest)
            went = False
            for s in slow:
                went |= self.step(s)
            n += 1
            if after is not None:
                went |= any([self.step(r) for r in rest])
            if not went and not self.settle(list(self.actors)):
                break
        stand = [a for a, at in self.at.items() if at != "end" and a not in ("copy", "pipe")]
        return not stand and not self.copies and not self.pipe, stand


def _roles(m):
    return [[a] for a in m.actors] + [[a for a in m.actors if a.startswith(p)] for p in ("mma", "dq0", "dq1", "epi")]


def _check(G, rings):
    for steps in (1, 2, 5, 23):
        for slow in _roles(Model(steps, G, rings)):
            for after in [None] + list(range(0, 3 * steps, 2)):
                ok, stand = Model(steps, G, rings).finish(slow, after)
                assert ok, "steps %d, %s held (%s): %s stand" % (steps, slow, after, stand)


@pytest.mark.parametrize("group", [32, 64, 128])
@pytest.mark.parametrize("S", [1, 33, 65, 100])
def test_every_role_comes_to_its_end_whichever_is_slow(S, group):
    tile, rings = pkg.shard_debug_gemm_rings(S, group)
    assert tile >= min(S, 64)
    _check(128 // group, rings)


@pytest.mark.parametrize("accumulators,G", [(8, 1), (6, 1), (5, 1)])
def test_the_model_stands_with_more_accumulators_than_completion_barriers(accumulators, G):
    _, rings = pkg.shard_debug_gemm_rings(64, 128 // G)
    rings[3] = accumulators
    with pytest.raises(AssertionError, match="stand"):
        _check(G, rings)

