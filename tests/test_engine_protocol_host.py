"""A model of the n = 4 engine's hand-offs (qcs_engine4.cu: jobs, rows, product
and sums of three sets), run under random interleavings of its warps on the
CPU.  The warps follow the kernel's control flow; every wait is for a phase
parity.  Checked on every schedule:
- every warp finishes, with any number of rounds per set, none included, and
  with rounds that have no W point (the MMA warp then arrives itself);
- no barrier runs two phases ahead of a warp that waits on it, so a parity
  wait cannot be taken for another phase's;
- what a warp reads is of its own round, and nothing is overwritten before
  its last reader is through (jobs, rows of B, D, column sums);
- where a control warp gives up, every wait that cannot end runs out, and the
  MMA warp leaves no product in flight.
"""
import random

import pytest

SETS = 3


class Barrier:
    def __init__(self, count):
        self.count, self.pending, self.phase, self.seen = count, count, 0, {}

    def arrive(self):
        assert self.pending > 0
        self.pending -= 1
        if not self.pending:
            self.phase, self.pending = self.phase + 1, self.count

    def wait(self, who, parity):
        """One wait: yields until the phase of this parity has completed.
        who: None where the caller follows the barrier's phases itself."""
        while self.phase % 2 == parity:
            if (yield ("wait", lambda: self.phase % 2 != parity)) == "out":
                return False
        if who is None:
            return True
        self.seen[who] = self.seen.get(who, 0) + 1
        assert self.phase - self.seen[who] in (0, 1), "a parity wait met another phase"
        return True


class Set:
    def __init__(self, workers):
        self.jobs, self.rows, self.prod, self.sums = Barrier(1), Barrier(workers), Barrier(1), Barrier(workers)
        self.round, self.done, self.nw = 0, False, 0  # round published last
        self.b = [0] * workers                         # round of each worker's rows
        self.d = self.flying = 0                       # round of D; product in flight
        self.part = [0] * workers
        self.read = [0] * workers                      # round whose job the worker has read


def worker(w, sets):
    live, ph, first, rnd = [True] * SETS, 0, True, 0
    while True:
        rnd += 1
        for x in range(SETS):
            s = sets[x]
            if live[x]:
                if not (yield from s.jobs.wait(("w", w), ph)):
                    return False
                live[x] = not s.done
            if live[x]:
                assert s.round == rnd and not s.flying, "rows under a product in flight"
                s.read[w] = s.b[w] = rnd
                yield ("run", None)
                s.rows.arrive()
            y = SETS - 1 if x == 0 else x - 1
            if not live[y] or (x == 0 and first):
                continue
            t, er = sets[y], rnd - 1 if x == 0 else rnd
            if not (yield from t.prod.wait(("w", w), ph ^ 1 if x == 0 else ph)):
                return False
            assert t.round == er and (t.nw == 0 or t.d == er), "sums of another round's product"
            t.part[w] = er
            yield ("run", None)
            t.sums.arrive()
        if not any(live):
            return True
        ph, first = ph ^ 1, False


def mma(sets, workers):
    live, ph, rnd = [True] * SETS, 0, 0
    while any(live):
        rnd += 1
        for x in range(SETS):
            s = sets[x]
            if not live[x]:
                continue
            ok = yield from s.jobs.wait("m", ph)
            if ok and s.done:
                live[x] = False
                continue
            ok = ok and (yield from s.rows.wait("m", ph))
            if not ok:
                for y in range(SETS):
                    if live[y]:
                        yield from sets[y].prod.wait(None, ph if y < x else ph ^ 1)
                assert not any(t.flying for t in sets), "a product in flight at the end"
                return False
            assert s.round == rnd and s.b == [rnd] * workers, "a product of another round's rows"
            if s.nw:
                assert s.flying == 0
                s.flying = rnd
            else:
                s.prod.arrive()
            yield ("run", None)
        ph ^= 1
    return True


def tensor_core(sets, state):
    """Completes products in the order of their issue, some time later."""
    while not state["end"]:
        flying = [s for s in sets if s.flying]
        if not flying:
            yield ("wait", lambda: state["end"] or any(s.flying for s in sets))
            continue
        s = flying[0]
        s.d, s.flying = s.flying, 0
        s.prod.arrive()
        yield ("run", None)
    return True


def control(x, sets, workers, rounds, gives_up, rng):
    s, ph = sets[x], 0
    for r in range(1, rounds + 1):
        # the last round's readers are through: workers with jobs and D, the MMA warp with nw and rows
        assert s.read == [r - 1] * workers and not s.flying
        s.round, s.nw = r, rng.randrange(3)
        yield ("run", None)
        s.jobs.arrive()
        if r == gives_up:
            return False
        if not (yield from s.sums.wait("c", ph)):
            return False
        assert s.part == [r] * workers, "sums of another round"
        ph ^= 1
        yield ("run", None)
    s.done = True
    s.jobs.arrive()
    return True


def run(seed, workers, rounds, gives_up=None):
    rng = random.Random(seed)
    sets, state = [Set(workers) for _ in range(SETS)], {"end": False}
    tasks = {("w", w): worker(w, sets) for w in range(workers)}
    tasks["m"] = mma(sets, workers)
    for x in range(SETS):
        tasks["c", x] = control(x, sets, workers, rounds[x], gives_up[1] if gives_up and gives_up[0] == x else 0, rng)
    tasks["t"] = tensor_core(sets, state)
    blocked, results, ran_out = {}, {}, set()
    while tasks:
        ready = [k for k in tasks if k not in blocked or blocked[k]()]
        if set(tasks) == {"t"}:
            state["end"] = True
            ready = ["t"]
        if ready:
            k, send = rng.choice(ready), None
        else:
            assert gives_up, "deadlock"
            # waits run out: the tensor core always gets on, so it is none of them
            k, send = rng.choice([k for k in tasks if k != "t"]), "out"
            ran_out.add(k)
        was_blocked = blocked.pop(k, None) is not None
        try:
            kind, pred = tasks[k].send(send if was_blocked else None)
            if kind == "wait":
                blocked[k] = pred
        except StopIteration as e:
            results[k] = e.value
            del tasks[k]
    return results, ran_out


@pytest.mark.parametrize("workers", [1, 2, 5])
def test_hand_offs_under_random_schedules(workers):
    for seed in range(250):
        rng = random.Random(1000 * workers + seed)
        rounds = [rng.choice([0, 0, 1, 2, 3, 7]) for _ in range(SETS)]
        results, _ = run(seed, workers, rounds)
        assert all(results.values()), (seed, rounds, results)


@pytest.mark.parametrize("workers", [1, 3])
def test_a_control_warp_that_gives_up_ends_the_run(workers):
    for seed in range(250):
        rng = random.Random(77 * workers + seed)
        rounds = [rng.randint(1, 6) for _ in range(SETS)]
        x = rng.randrange(SETS)
        results, ran_out = run(seed, workers, rounds, gives_up=(x, rng.randint(1, rounds[x])))
        # the CTA's answer is the conjunction over its warps
        assert not results["c", x] and not results["m"] and "t" not in ran_out, (seed, rounds)
