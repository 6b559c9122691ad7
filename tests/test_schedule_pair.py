"""Host-side checks of the CTA-pair variant's schedule (emul_schedule_pair; no
GPU needed): every kept slice pair and K chunk is summed exactly once within
the exact-accumulation budget, the last job is the final one and of level 2,
the staged planes fit, and the state's bounds hold in exact integers with and
without the low bits put aside."""
import pytest

from paper_2509_23565_gb300 import binding

KBK, BUDGET = 32, 1040
KS = (1, 31, 33, 128, 130, 256, 1024, 1056, 2080, 4096, 16384, 65536)
SETS = [(s, s, 0) for s in range(1, 9)] + [(7, 7, 9), (7, 7, 14), (3, 3, 6), (8, 8, 4), (3, 7, 0), (8, 2, 0), (5, 8, 9)]


@pytest.mark.parametrize("sa,sb,t", SETS)
def test_pair_schedule(sa, sb, t):
    s, tt = max(sa, sb), t or max(sa, sb) + 1
    for k in KS:
        got = binding.schedule_pair(sa, sb, k, t)
        if got is None:
            # at the method's own threshold only 8 slices beyond k = 16384 (2^63 k > 2^(61+16)) go without
            assert t != 0 or (s == 8 and k > 16384), (sa, sb, k)
            continue
        sweeps, kind, stash = got
        nch = (k + KBK - 1) // KBK
        seen, jobs = {}, []
        for w in sweeps:
            assert 1 <= len(w["jobs"]) <= 4 and w["kcs"] >= 1 and w["kcs"] * w["nplanes"] <= s
            for j, (L, pb, pe) in enumerate(w["jobs"]):
                assert (pe - pb + 1) * (w["k1c"] - w["k0c"]) * KBK <= BUDGET
                for p in range(pb, pe + 1):
                    assert 1 <= p <= sa and 1 <= L - p <= sb and max(p, L - p) <= w["nplanes"]
                    seen.setdefault((p, L - p), []).append((w["k0c"], w["k1c"]))
                jobs.append((L, pe - pb + 1, w["k1c"] - w["k0c"], w["final"] == j))
        want = {(p, q) for p in range(1, sa + 1) for q in range(1, sb + 1) if p + q <= tt}
        assert set(seen) == want
        for r in seen.values():          # the chunk ranges tile [0, nch)
            r.sort()
            assert r[0][0] == 0 and r[-1][1] == nch and all(a[1] == b[0] for a, b in zip(r, r[1:]))
        assert [j[3] for j in jobs] == [False] * (len(jobs) - 1) + [True] and jobs[-1][0] == 2
        # worst-case magnitude of the state before the final job's term
        R, units = 0, 0
        for i, (L, n, c, fin) in enumerate(jobs):
            w = 7 * (tt - L) - units
            assert w >= 0
            if fin:
                assert (n * c * KBK * 127 ** 2 << w) < 2 ** 62 or kind == 1
                break
            R += n * c * KBK * 127 ** 2 << w
            assert R < 2 ** 61
            if i == stash:
                assert kind == 2
                R, units = (R >> 16) + 1, 16
        assert (stash >= 0) == (kind == 2)
