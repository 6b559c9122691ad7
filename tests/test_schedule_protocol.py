"""The product kernel's barrier protocol on its schedules, simulated on the host
(no GPU needed).

One tile loop per role, as in the kernel: a producer fills ring stages; two
issuing warps take a sweep's jobs alternately, wait for a stage to be full, for a
job's TMEM slot before the job's first MMA, commit the slot after the job's last
one and free the stage together; the epilogue waits for each job in order, two
adjacent levels of a sweep in one step, and releases the slots.  Job i, counted over
all tiles, has slot i % 4 and waits on the parities of i / 4.  Every barrier is an
mbarrier: a wait on parity p passes once the phase of parity p that the barrier is
in, or has just left, is complete, so a wrong count passes too early or never.
"""
import pytest

from paper_2509_23565_gb300 import binding

KS = (1, 100, 256, 300, 1000, 1056, 2080)
ST = [(1, 2), (2, 3), (3, 4), (5, 6), (6, 7), (7, 8), (8, 9), (7, 2), (7, 14), (8, 16), (4, 6)]


class Barrier:
    def __init__(self, count):
        self.count, self.pending, self.phase = count, count, 0

    def arrive(self):
        self.pending -= 1
        assert self.pending >= 0
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1

    def passed(self, parity):                # the kernel's try_wait.parity
        return self.phase & 1 != parity


def one_cta(s, t, k):
    out = []
    for wide in (False, True):
        r = binding.schedule(s, k, wide=wide, t=t)
        if r is not None:
            out.append([(w["k0c"], w["k1c"], w["kcs"], [(w["L0"], bool(w["flags0"]))]
                         + ([(w["L1"], bool(w["flags1"]))] if w["L1"] else [])) for w in r[0]])
    return out


def pairs(s, t, k):
    r = binding.schedule_pair(s, s, k, t)
    return [] if r is None else [[(w["k0c"], w["k1c"], w["kcs"], [(j[0], w["final"] == i) for i, j in enumerate(w["jobs"])])
                                  for w in r[0]]]


def together(jobs, j, paired):
    """Jobs j and j + 1 of a sweep are drained in one step (not by the 128-bit state)."""
    return (paired and j + 1 < len(jobs) and abs(jobs[j + 1][0] - jobs[j][0]) == 1
            and not jobs[j][1] and not jobs[j + 1][1])


def simulate(sweeps, stages, tiles, paired, slot_of=lambda i: i % 4, parity_of=lambda i: i // 4 & 1, sync_stage=True):
    """Runs the four roles, the ones that can go on in an order that favours one
    of them, to the end; asserts on a deadlock, a slot taken while it is in use, a
    job drained before it is complete and a stage refilled while it is read."""
    for favoured in range(4):
        full, empty = [Barrier(1) for _ in range(stages)], [Barrier(2 if sync_stage else 1) for _ in range(stages)]
        sfull, sempty = [Barrier(1) for _ in range(4)], [Barrier(1) for _ in range(4)]
        owner, done = [None] * 4, [False] * 4
        readers = [set() for _ in range(stages)]

        def fills():
            for _ in range(tiles):
                for (k0, k1, kcs, jobs) in sweeps:
                    yield from ((jobs, kc == k0, kc + kcs >= k1) for kc in range(k0, k1, kcs))

        def producer():
            for f, _ in enumerate(fills()):
                st, par = f % stages, (f // stages & 1) ^ 1
                while not empty[st].passed(par):
                    yield False
                assert not readers[st], "stage refilled while it is read"
                readers[st] = {0, 1}
                full[st].arrive()
                yield True

        def issuer(w):
            job0 = 0
            for f, (jobs, first, last) in enumerate(fills()):
                st, par = f % stages, f // stages & 1
                while not full[st].passed(par):
                    yield False
                assert w in readers[st], "stage read before it is filled"
                for j in range(w, len(jobs), 2):
                    i = job0 + j
                    sl = slot_of(i)
                    if first:
                        while not sempty[sl].passed(parity_of(i) ^ 1):
                            yield False
                        assert owner[sl] is None, "slot taken while it is in use"
                        owner[sl], done[sl] = i, False
                    assert owner[sl] == i
                    if last:
                        done[sl] = True
                        sfull[sl].arrive()
                    yield True
                readers[st].discard(w)
                if sync_stage or w == 0:
                    empty[st].arrive()
                if last:
                    job0 += len(jobs)
                yield True

        def epilogue():
            i = 0
            for _ in range(tiles):
                for (_, _, _, jobs) in sweeps:
                    j = 0
                    while j < len(jobs):
                        n = 2 if together(jobs, j, paired) else 1
                        for q in range(i, i + n):
                            while not sfull[slot_of(q)].passed(parity_of(q)):
                                yield False
                            assert owner[slot_of(q)] == q and done[slot_of(q)], "job drained before it is complete"
                        yield True
                        for q in range(i, i + n):
                            owner[slot_of(q)] = None
                            sempty[slot_of(q)].arrive()
                        i, j = i + n, j + n
                        yield True

        roles = {0: producer(), 1: issuer(0), 2: issuer(1), 3: epilogue()}
        order = [favoured] + [r for r in range(4) if r != favoured]
        while roles:
            for r in [r for r in order if r in roles]:
                step = next(roles[r], None)
                if step is None:
                    del roles[r]
                if step or step is None:
                    break
            else:
                raise AssertionError("deadlock")


@pytest.mark.parametrize("s,t", ST)
@pytest.mark.parametrize("kind", ["one CTA", "pair"])
def test_protocol(s, t, kind):
    for k in KS:
        for sweeps in one_cta(s, t, k) if kind == "one CTA" else pairs(s, t, k):
            wide = kind == "one CTA" and not any(fin for w in sweeps for (_, fin) in w[3])
            for stages in (2, 5):
                simulate(sweeps, stages, 3, paired=not wide)
                simulate(sweeps, stages, 3, paired=False)        # level sums: every job on its own


@pytest.mark.parametrize("wrong", ["parity", "slots", "stage"])
def test_the_simulation_sees_a_wrong_rule(wrong):
    """The same roles with a parity that never changes, three slots used as four, or
    stages freed by one issuing warp alone do not run to the end."""
    sweeps = pairs(7, 8, 256)[0]
    with pytest.raises(AssertionError):
        if wrong == "parity":
            simulate(sweeps, 2, 3, True, parity_of=lambda i: 0)
        elif wrong == "slots":
            simulate(sweeps, 2, 3, True, slot_of=lambda i: i % 3)
        else:
            simulate(sweeps, 2, 3, True, sync_stage=False)
