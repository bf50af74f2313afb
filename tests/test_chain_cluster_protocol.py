"""Host model of the hand-overs of the FP64 cluster step (no GPU).

A chain runs on a cluster of G CTAs of four warps.  CTA r owns the bonds and modes
r S .. r S + S - 1 (S = ceil(M / G)), its warps one each in turn; with M < G S the last
CTA has fewer and CTAs past it have none.  Per step every warp sends the forces v of its
bonds, waits until all M have arrived, and sends its modes R in the same way.  A value is
an asynchronous store that counts its bytes on the reader's mbarrier, whose count thread 0
arms for the next phase once the last one is over.

The warps run as coroutines under random interleavings, stores arrive late and out of
order, and every run checks
  * no deadlock (a barrier whose bytes ran past its count never completes);
  * every parity wait is for the barrier's current phase or the one before it;
  * no value is overwritten before every warp of that CTA has read it, and every value
    that a warp reads is this step's;
  * after a timeout (one CTA sends nothing, every wait that can no longer be met gives up)
    all warps come to the end and no barrier is armed in a phase that is not over.
Negative controls: values sent to CTAs that own nothing, on which nobody waits, and warps
that own nothing waiting on the barriers, and counts armed after a timeout must be caught."""
import random

import pytest

WARPS = 4


class ProtocolError(Exception):
    pass


class Barrier:
    """One arrival (the armed count) and its transaction bytes per phase."""

    def __init__(self, name):
        self.name, self.pending, self.tx, self.phase = name, 1, 0, 0

    def _complete(self):
        if self.pending == 0 and self.tx == 0:
            self.phase, self.pending = self.phase + 1, 1

    def arm(self, n):
        if self.pending != 1:
            raise ProtocolError(f"{self.name}: armed twice in phase {self.phase}")
        self.pending, self.tx = 0, self.tx + n
        self._complete()

    def count(self, n):
        self.tx -= n            # may go below zero before the count is armed
        self._complete()


class Cluster:
    def __init__(self, M, G, steps, seed, idle_ctas=False, idle_warps=False, stall=None, arm_always=False):
        """idle_ctas: CTAs that own nothing receive every value and run the steps;
        idle_warps: warps that own nothing wait on the barriers; stall: a CTA that gave
        up before its first step; arm_always: counts are armed after a timeout too."""
        self.M, self.G, self.steps = M, G, steps
        self.rng = random.Random(seed)
        self.lag = (None, 0.2, 0.05)[seed % 3]          # how eagerly stores arrive
        self.idle_ctas, self.idle_warps = idle_ctas, idle_warps
        self.stall, self.arm_always = stall, arm_always
        S = (M + G - 1) // G
        self.own = [list(range(min(M, r * S), min(M, r * S + S))) for r in range(G)]
        self.ctas = [r for r in range(G) if self.own[r] or idle_ctas]
        self.bar = {(r, a): Barrier(f"{r}.{a}") for r in range(G) for a in "vR"}
        self.val = {(r, a): [-1] * M for r in range(G) for a in "vR"}   # step of each value held
        for r in range(G):
            self.val[r, "R"] = [0] * M                  # the state of step 0
        self.read = {}                                  # (cta, array, warp) -> steps read
        self.stores = []
        self.met = {r: [0] * WARPS for r in range(G)}   # block barriers reached
        for r in range(G):
            self.bar[r, "v"].arm(M)
            self.bar[r, "R"].arm(M - 1)

    def mine(self, r, w):
        return self.own[r][w::WARPS]

    def reads(self, r, w, a):
        # mode 0, the centre of mass, takes no force and is not sent
        return bool([p for p in self.mine(r, w) if a == "R" or p])

    def send(self, r, a, i, step):
        for q in self.ctas:
            self.stores.append((q, a, i, step))

    def land(self, k):
        q, a, i, step = self.stores.pop(k)
        last = step - 1
        for w in range(WARPS):
            if self.reads(q, w, a) and self.read.get((q, a, w), -1) < last:
                raise ProtocolError(f"CTA {q}: {a}_{i} of step {step} lands before warp {w} has read step {last}")
        self.val[q, a][i] = step
        self.bar[q, a].count(1)

    def wait(self, r, a, x):
        bar = self.bar[r, a]

        def done():
            if (bar.phase & 1) == (x & 1):              # the phase of this parity is under way
                if bar.phase > x:
                    raise ProtocolError(f"{bar.name} at phase {bar.phase}: a wait for phase {x} would hang")
                return False
            if bar.phase != x + 1:
                raise ProtocolError(f"{bar.name} at phase {bar.phase}: a wait for phase {x} would pass")
            return True
        return done

    def take(self, r, w, a, step):
        if not self.reads(r, w, a):
            return
        skip = 1 if a == "R" else 0
        if any(t != step for t in self.val[r, a][skip:]):
            raise ProtocolError(f"CTA {r} warp {w}: {a} of step {step} reads {self.val[r, a]}")
        self.read[r, a, w] = step

    def warp(self, r, w):
        mine = self.mine(r, w)
        waits = bool(mine) or self.idle_warps or (self.idle_ctas and not self.own[r])
        if not self.own[r] and not self.idle_ctas:
            return
        ok = r != self.stall
        for s in range(self.steps):
            if ok:
                self.take(r, w, "R", s)
            yield None
            for n in mine if ok else []:
                self.send(r, "v", n, s)
            self.met[r][w] += 1
            yield lambda: min(self.met[r]) >= s + 1
            if waits and ok:
                ok = yield self.wait(r, "v", s)
            if w == 0 and (ok or self.arm_always):
                self.bar[r, "v"].arm(self.M)
            yield None
            if ok:
                self.take(r, w, "v", s)
            for p in mine if ok else []:
                if p:
                    self.send(r, "R", p, s + 1)
            yield None
            if waits and ok:
                ok = yield self.wait(r, "R", s)
            if w == 0 and (ok or self.arm_always):
                self.bar[r, "R"].arm(self.M - 1)
            yield None

    def run(self):
        roles = [[self.warp(r, w), None, False, False] for r in range(self.G) for w in range(WARPS)]
        # some warps run more often than others, those that own nothing seldom
        weight = [self.rng.choice((1, 1, 8)) if self.mine(r, w) else 0.02 for r in range(self.G) for w in range(WARPS)]
        while True:
            ready = [i for i, (g, cond, done, _) in enumerate(roles) if not done and (cond is None or cond())]
            if self.stores and (not ready or self.lag is None or self.rng.random() < self.lag):
                self.land(self.rng.randrange(len(self.stores)))
                continue
            met = bool(ready)
            if not ready:
                if all(x[2] for x in roles):
                    return
                # the barriers of a block's warps are not bounded; what waits on the others gives up
                ready = [i for i, (g, cond, done, _) in enumerate(roles) if not done and cond.__name__ == "done"]
                if self.stall is None or not ready:
                    raise ProtocolError("deadlock")
            i = self.rng.choices(ready, [weight[k] for k in ready])[0]
            try:
                roles[i][1] = roles[i][0].send(met if roles[i][3] else None)
                roles[i][3] = True
            except StopIteration:
                roles[i][2] = True


# (M, G): fewer beads than CTAs, CTAs without any, warps without any, all in use, uneven last CTA
SHAPES = [(3, 8), (7, 16), (17, 16), (20, 16), (20, 8), (100, 16), (64, 16), (65, 16)]


@pytest.mark.parametrize("M,G", SHAPES)
def test_hand_overs_under_random_interleavings(M, G):
    for seed in range(6 if M > 30 else 30):
        Cluster(M, G, 4, seed).run()


def caught(M, G, seeds, **kw):
    n = 0
    for seed in range(seeds):
        try:
            Cluster(M, G, 6, seed, **kw).run()
        except ProtocolError:
            n += 1
    return n


@pytest.mark.parametrize("M,G", [(7, 16), (20, 16), (17, 16), (100, 16)])
def test_sending_to_ctas_that_own_nothing_is_caught(M, G):
    assert caught(M, G, 20, idle_ctas=True) > 0


@pytest.mark.parametrize("M,G", [(3, 8), (20, 16)])
def test_waits_of_warps_that_own_nothing_are_caught(M, G):
    assert caught(M, G, 40, idle_warps=True) > 0


@pytest.mark.parametrize("M,G", [(20, 16), (64, 16), (20, 8)])
def test_every_warp_comes_to_the_end_after_a_timeout(M, G):
    for seed in range(10):
        Cluster(M, G, 4, seed, stall=(M - 1) // ((M + G - 1) // G)).run()
        with pytest.raises(ProtocolError, match="armed twice"):
            Cluster(M, G, 4, seed, stall=0, arm_always=True).run()


def update_lanes(rng, ordered, shear):
    """The 24 lanes of a warp that update one mode: lane 8 a + j reads R of its axis (axis 0
    with shear also that of axis 1); one lane of each axis then stores the new value in this
    CTA's own copy.  Lanes run in any order after the last shuffle; `ordered`: a warp barrier
    lies between the reads and the stores.  Returns the axes that a lane read too late."""
    new, late, order = set(), set(), [(a, j) for a in range(3) for j in range(8)]
    rng.shuffle(order)

    def read(a):
        late.update(({a, 1} if shear and a == 0 else {a}) & new)

    if ordered:
        for a, _ in order:
            read(a)
    for a, j in order:
        if not ordered:
            read(a)
        if j == 3:
            new.add(a)
    return late


@pytest.mark.parametrize("shear", [False, True])
def test_a_mode_is_read_by_all_lanes_before_it_is_overwritten(shear):
    for seed in range(20):
        assert not update_lanes(random.Random(seed), True, shear)
        assert update_lanes(random.Random(seed), False, shear)      # negative control
