"""Host model of the hand-overs of the 512-bead lane step (no GPU).

A tile runs on a cluster of two CTAs, a parity of the modes each.  Per step and CTA:
  work warps  wait for the inverse MMAs, send the other CTA's bond vectors into its U, wait
              for theirs, put their forces into operand X of both CTAs, wait for the forward
              MMAs, update the modes and put them into X;
  MMA warps   (two, one accumulator each) inverse from X, two chunks of normals, forward
              from X, the other two chunks; what they read is free when its commit lands;
  noise warps draw every second chunk into their CTA's buffer of both CTAs once four commits
              (both CTAs, both MMA warps) have freed it;
  warp 19     reads the centre of mass's increments and arms the next step's counts.
What crosses between the CTAs are asynchronous stores that count on the reader's mbarrier;
they land late and in any order here, and may land before the count is armed.  MMAs retire
in order per warp; a commit to the other CTA lands late too.  Every run checks
  * no deadlock, no arrival past a barrier's count;
  * every parity wait is for the barrier's current phase or the one before it;
  * X, U, the noise buffers and the increments are not overwritten before their readers are
    done, and every reader finds its own step's content;
  * nothing is in flight when both CTAs have come to the end.
Negative controls: noise warps that do not wait for a free buffer, noise warps that leave
without waiting for the last commits, and a warp 19 that arms the first step's counts before
it has seen the first modes (and can then be two phases behind), must be caught."""
import random

import pytest


class ProtocolError(Exception):
    pass


class Barrier:
    def __init__(self, name, count):
        self.name, self.count, self.pending, self.tx, self.phase = name, count, count, 0, 0

    def _complete(self):
        if self.pending < 0:
            raise ProtocolError(f"{self.name}: more arrivals than phase {self.phase} counts")
        if self.pending == 0 and self.tx == 0:
            self.phase, self.pending = self.phase + 1, self.count

    def arrive(self, tx=0):
        self.pending, self.tx = self.pending - 1, self.tx + tx
        self._complete()

    def land(self):
        self.tx -= 1
        self._complete()


class Pair:
    NOISE = 2           # noise warps

    def __init__(self, batches, steps, seed, free_wait=True, last_wait=True, wait_first=True):
        """batches: of each work warp (some have none)."""
        self.batches, self.steps = batches, steps
        self.free_wait, self.last_wait, self.wait_first = free_wait, last_wait, wait_first
        self.nb = sum(map(len, batches))
        self.rng = random.Random(seed)
        self.lag = (None, 0.3, 0.05)[seed % 3]          # how eagerly asynchronous work gets on ...
        self.drift = (1.0, 0.02)[seed // 3 % 2]         # ... and what crosses between the CTAs
        self.bar, self.at = {}, {}      # at: (cta, place) -> [tag, readers left]
        for r in range(2):
            for k, n in (("r_ready", len(batches)), ("v_ready", len(batches) + 1), ("u_in", 1), ("u_done", 2),
                         ("inc_done", 2), ("n_ready", self.NOISE), ("n_other", 1), ("n_free", 4)):
                self.bar[r, k] = Barrier(f"{r}.{k}", n)
            for b in range(self.nb):
                for half in range(2):
                    self.at[r, "X", b, half] = [None, set()]
        self.flight = []                # (description, action)
        self.pipe = {(r, e): [] for r in range(2) for e in range(2)}

    def put(self, key, tag, readers):
        cur = self.at.get(key, [None, set()])
        if cur[1]:
            raise ProtocolError(f"{key}: {tag} over {cur[0]}, still read by {cur[1]}")
        self.at[key] = [tag, set(readers)]

    def take(self, key, tag, who):
        cur = self.at.get(key)
        if not cur or cur[0] != tag or who not in cur[1]:
            raise ProtocolError(f"{key}: {who} wants {tag}, finds {cur}")
        cur[1].discard(who)

    def send(self, key, tag, readers, bar):
        def act():
            self.put(key, tag, readers)
            self.bar[bar].land()
        self.flight.append((f"{tag} to {key}", act))

    def wait(self, r, k, x):
        bar = self.bar[r, k]

        def done():
            if (bar.phase & 1) == (x & 1):
                if bar.phase > x:
                    raise ProtocolError(f"{bar.name} at phase {bar.phase}: a wait for phase {x} would hang")
                return False
            if bar.phase != x + 1:
                raise ProtocolError(f"{bar.name} at phase {bar.phase}: a wait for phase {x} would pass")
            return True
        return done

    def put_modes(self, r, mine, sp):
        for b in mine:
            for half in range(2):
                self.put((r, "X", b, half), ("R", sp), {0, 1})
        self.bar[r, "r_ready"].arrive()

    def work(self, r, w):
        mine, p = self.batches[w], r ^ 1
        self.put_modes(r, mine, 0)
        for sp in range(self.steps):
            yield self.wait(r, "u_done", sp)
            for b in mine:
                self.send((p, "U", b), ("U", sp), {"work"}, (p, "u_in"))
                yield None
            yield self.wait(r, "u_in", sp)
            held = []
            for i, b in enumerate(mine):
                self.take((r, "U", b), ("U", sp), "work")
                self.put((r, "X", b, r), ("V", sp), {0, 1})
                held.append(b)
                if i != 0 or len(mine) == 1:        # the first batch's goes with the second's
                    for h in held:
                        self.send((p, "X", h, r), ("V", sp), {0, 1}, (p, "v_ready"))
                    held = []
                yield None
            self.bar[r, "v_ready"].arrive()
            yield self.wait(r, "inc_done", sp)
            if w == 0:
                self.put((r, "d0"), sp, {"cm"})
            self.put_modes(r, mine, sp + 1)
            yield None

    def mma(self, r, e):
        pipe, seq = self.pipe[r, e], 0

        def x(tag):
            pipe.append(("read", [(r, "X", b, h) for b in range(self.nb) for h in range(2)], tag))

        def chunk(ch):
            nonlocal seq
            own = ch % 2 == r
            yield self.wait(r, "n_ready" if own else "n_other", seq // 2)
            if e == 0 and not own:
                self.bar[r, "n_other"].arrive(tx=self.NOISE)
            pipe.append(("read", [(r, "Z", ch % 2, n) for n in range(self.NOISE)], ("Z", seq)))
            pipe.append(("commit", (ch % 2, "n_free")))
            seq += 1

        if e == 0:
            self.bar[r, "n_other"].arrive(tx=self.NOISE)
        for sp in range(self.steps):
            yield self.wait(r, "r_ready", sp)
            x(("R", sp))
            pipe.append(("commit", (r, "u_done")))
            yield None
            for ch in range(2):
                yield from chunk(ch)
            yield self.wait(r, "v_ready", sp)
            x(("V", sp))
            yield None
            for ch in range(2, 4):
                yield from chunk(ch)
            pipe.append(("commit", (r, "inc_done")))

    def noise(self, r, n):
        total = 2 * self.steps
        for q in range(total):
            if q and self.free_wait:
                yield self.wait(r, "n_free", q - 1)
            seq = 2 * q + r
            self.put((r, "Z", r, n), ("Z", seq), {0, 1})
            self.send((r ^ 1, "Z", r, n), ("Z", seq), {0, 1}, (r ^ 1, "n_other"))
            self.bar[r, "n_ready"].arrive()
            yield None
        if self.last_wait:
            yield self.wait(r, "n_free", total - 1)

    def centre(self, r):
        def arm():
            self.bar[r, "u_in"].arrive(tx=self.nb)
            self.bar[r, "v_ready"].arrive(tx=self.nb)
        if not self.wait_first:
            arm()
        yield self.wait(r, "r_ready", 0)
        if self.wait_first:
            arm()
        for sp in range(self.steps):
            yield self.wait(r, "r_ready", sp + 1)
            self.take((r, "d0"), sp, "cm")
            if sp + 1 < self.steps:
                arm()
            yield None

    def retire(self, r, e):
        item = self.pipe[r, e].pop(0)
        if item[0] == "read":
            for key in item[1]:
                self.take(key, item[2], e)
        elif item[1][0] == r:
            self.bar[item[1]].arrive()
        else:                           # the other CTA's barrier: on its way
            self.flight.append((f"commit to {item[1]}", lambda k=item[1]: self.bar[k].arrive()))

    def run(self):
        roles = [[g, None, False] for r in range(2) for g in
                 [self.work(r, w) for w in range(len(self.batches))] + [self.mma(r, e) for e in range(2)] +
                 [self.noise(r, n) for n in range(self.NOISE)] + [self.centre(r)]]
        weight = [self.rng.choice((1, 1, 8, 0.1)) for _ in roles]
        weight[-1] = self.rng.choice((1, 0.01))         # a warp 19 may run seldom
        while True:
            ready = [i for i, (g, cond, done) in enumerate(roles) if not done and (cond is None or cond())]
            late = [("store", i) for i in range(len(self.flight))] + [("pipe", k) for k, v in self.pipe.items() if v]
            if all(x[2] for x in roles):
                if late:
                    raise ProtocolError("the CTAs leave with stores or commits in flight")
                return
            if late and (not ready or self.lag is None or self.rng.random() < self.lag):
                kind, i = self.rng.choices(late, [self.drift if x[0] == "store" else 1.0 for x in late])[0]
                if kind == "store":
                    self.flight.pop(i)[1]()
                else:
                    self.retire(*i)
                continue
            if not ready:
                raise ProtocolError("deadlock")
            i = self.rng.choices(ready, [weight[k] for k in ready])[0]
            try:
                roles[i][1] = next(roles[i][0])
            except StopIteration:
                roles[i][2] = True


# batches of the work warps: one in all, one each, uneven, three of the largest tile's warps
BATCHES = [[[0], []], [[0], [1]], [[0, 2], [1], []], [[0, 2, 4], [1, 3, 5]]]


@pytest.mark.parametrize("batches", BATCHES, ids=["one", "two", "uneven", "full"])
@pytest.mark.parametrize("steps", [1, 2, 4])
def test_hand_overs_under_random_interleavings(batches, steps):
    for seed in range(60):
        Pair(batches, steps, seed).run()


@pytest.mark.parametrize("control", ["free_wait", "last_wait", "wait_first"])
def test_missing_waits_are_caught(control):
    caught = 0
    for seed in range(120):
        try:
            Pair([[0, 2], [1], []], 1, seed, **{control: False}).run()
        except ProtocolError:
            caught += 1
    assert caught > 0
