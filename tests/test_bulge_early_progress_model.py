"""CPU model of the bulge chase's progress rule (csrc/bulge.cu).  No GPU.

Sweep s publishes progress t+2 once its task t has stored everything AND the reflector of task t+1 has
been formed and its one band entry (beta) stored; task (s+1, t) loads its blocks once progress[s] >= t+3.
So the events of sweep s, in its own program order, are
    first reflector | task 0 | beta of task 1 | signal 2 | task 1 | beta of task 2 | signal 3 | ...
(beta of task t+1 is stored concurrently with the stores of task t; both precede signal t+2, and the loads
of task t+1 may run before or after it).  The model lists the band cells of each event, closes the order
"program order within a sweep" and "signal -> load" transitively, and checks that conflicting accesses of
different sweeps are ordered, in the direction that the sequential sweeps have."""
import numpy as np
import pytest


def events(n, b):
    """Per sweep: a list of (kind, t, [(is_write, r0, r1, c0, c1)]); kinds "load", "store", "beta", "signal", "end"."""
    out = []
    for s in range(0, n - 2):
        ev = []
        ln0 = min(b, n - s - 1)
        ev.append(("first", 0, [(False, s + 1, s + 1 + ln0, s, s + 1), (True, s + 1, s + 1 + ln0, s, s + 1)]))
        t = 0
        while True:
            p = s + 1 + t * b
            ln = min(b, n - p)
            p2 = p + ln
            ln2 = min(b, n - p2)
            pn = p + b
            lnn = min(b, n - pn) if pn < n else 0
            ev.append(("load", t, [(False, p, p + ln, p, p + ln), (False, p2, p2 + ln2, p, p + ln)]))
            st = [(True, p, p + ln, p, p + ln)]
            if t > 0:  # the bulge block L; its entry (p, p - b) was stored with the reflector
                st += [(True, p, p + ln, p - b + 1, p), (True, p + 1, p + ln, p - b, p - b + 1)]
            if lnn > 1:
                ev.append(("store", t, st + [(True, pn, pn + 1, p, p + 1)]))
                ev.append(("signal", t + 2, []))
                t += 1
                continue
            ev.append(("store", t, st))
            if lnn == 1:
                ev.append(("last", t + 1, [(True, pn, pn + 1, pn - b, pn)]))
            ev.append(("end", 0, []))
            break
        out.append(ev)
    return out


def overlap(a, c):
    r0, r1 = max(a[1], c[1]), min(a[2], c[2])
    c0, c1 = max(a[3], c[3]), min(a[4], c[4])
    return r0 < r1 and c0 < c1 and r1 - 1 >= c0


def known(ev_prev, need):
    """Index of the first event of the previous sweep that publishes progress >= need."""
    for i, (k, t, _) in enumerate(ev_prev):
        if (k == "signal" and t >= need) or k == "end":
            return i
    raise AssertionError


@pytest.mark.parametrize("n,b", [(3, 16), (5, 16), (20, 16), (33, 16), (67, 16), (100, 16), (40, 32), (97, 32),
                                 (130, 32), (70, 64), (150, 64)])
def test_every_conflict_is_ordered(n, b):
    evs = events(n, b)
    # bound[s][i][s1] = number of events of sweep s1 < s known complete when event i of sweep s starts
    bound = []
    checked = 0
    for s, ev in enumerate(evs):
        rows = []
        cur = np.zeros(s, dtype=np.int64)
        for i, (kind, t, acc) in enumerate(ev):
            if s > 0 and kind in ("first", "load", "last"):
                need = 3 if kind == "first" else t + 3
                j = known(evs[s - 1], need)
                new = np.zeros(s, dtype=np.int64)
                new[s - 1] = j
                if s > 1:
                    # what the events of sweep s-1 up to j knew (its signal follows its own program order)
                    new[: s - 1] = bound[s - 1][j]
                cur = np.maximum(cur, new)
            rows.append(cur.copy())
        bound.append(rows)
    for s, ev in enumerate(evs):
        for i, (kind, t, acc) in enumerate(ev):
            for s1 in range(max(0, s - 2 * b), s):
                done = bound[s][i][s1]
                for i1, (k1, t1, acc1) in enumerate(evs[s1]):
                    if i1 < done:
                        continue
                    for a in acc:
                        for c in acc1:
                            if (a[0] or c[0]) and overlap(a, c):
                                raise AssertionError((s, kind, t, a, s1, k1, t1, c))
                    checked += 1
    assert n < 20 or checked > 0


def test_signalling_before_the_next_reflector_is_caught():
    """Without the beta of task t+2 the load of (s+1, t) would read an entry that is still to change."""
    n, b = 60, 16
    evs = events(n, b)
    s = 0
    load0 = next(e for e in evs[s + 1] if e[0] == "load" and e[1] == 0)
    store1 = next(e for e in evs[s] if e[0] == "store" and e[1] == 1)
    beta2 = store1[2][-1]
    assert any(overlap(a, beta2) for a in load0[2])
