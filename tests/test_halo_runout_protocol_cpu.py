"""The halo hand-over of the register/tile chain on clusters when a wait runs
out, as a CPU model under random interleavings.

At hand-over n the threads that own a CTA's outermost pair rows send them to
the neighbours' slots of parity n mod 2 (st.async: the bytes, landing at any
later time, count on the neighbour's mbarrier of that side and parity); the
threads that hold halo rows wait, at most a limit, for their side's barrier,
one of them arms it again for hand-over n + 2, and a CTA barrier closes the
hand-over.  Where a thread's run is shorter than the halo and the outermost
rows together, the threads that send are not the ones that receive.

The model lets any wait run out at any time and checks that no byte is counted
on a phase that is not armed for its hand-over (an unarmed barrier's
transaction count would fall without bound) and that none lands in a CTA that
has left.  The protocol of one flag per thread, cleared where that thread's own
wait ran out, and of a drain of the lost phase alone fails both."""
import random

import pytest


class Side:
    """The two barriers (by parity) of one side of one CTA."""

    def __init__(self):
        self.armed = [0, 1]  # the hand-over each parity's open phase is armed for
        self.got = {}        # hand-over -> rows landed
        self.done = set()    # hand-overs whose phase has completed

    def land(self, n, rows):
        assert self.armed[n & 1] == n, f"bytes of hand-over {n} on a phase that is not armed for it"
        self.got[n] = self.got.get(n, 0) + 1
        if self.got[n] == rows:
            self.done.add(n)
            self.armed[n & 1] = None


def roles(R, TY, D):
    """Threads of a column by what they do: runs of R pair rows, TY a column, D halo rows a side."""
    own = TY * R - 2 * D
    out = []
    for ty in range(TY):
        rows = range(ty * R, ty * R + R)
        out.append({"recv": [any(f < D for f in rows), any(f >= D + own for f in rows)],
                    "send": [sum(D <= f < 2 * D for f in rows), sum(own <= f < own + D for f in rows)]})
    return out


def run(C, shape, H, seed, protocol, limit):
    """One random schedule of H hand-overs on C CTAs; a wait that cannot go on
    runs out with probability `limit`.  None, or what went wrong."""
    rng = random.Random(seed)
    D, TY = shape[2], shape[1]
    role = roles(*shape)
    sides = [[Side(), Side()] for _ in range(C)]  # 0: filled by the CTA below, 1: by the one above
    flight = []                                   # (CTA, side, hand-over)
    gone = [False] * C
    lost = [False] * C                            # the CTA's flag
    lost_at = [[None] * TY for _ in range(C)]     # hand-over each thread's own wait ran out at
    th = {(c, t): {"n": 0, "st": "send", "side": 0, "drain": None} for c in range(C) for t in range(TY)}
    met = {}

    def has(c, side):
        return c > 0 if side == 0 else c + 1 < C

    def stopped(c, t):
        return lost[c] if protocol == "cta" else lost_at[c][t] is not None

    def meet(key, t, size):
        met.setdefault(key, set()).add(t)
        return len(met[key]) == size

    steps, speed = 0, rng.choice((0.3, 0.005))  # of the bytes on their way
    while any(s["st"] != "left" for s in th.values()) or flight:
        steps += 1
        if steps > 200000:
            return "no end"
        if flight and rng.random() < speed:
            c, side, n = flight.pop(rng.randrange(len(flight)))
            if gone[c]:
                return f"bytes of hand-over {n} land in CTA {c} after it has left"
            try:
                sides[c][side].land(n, D)
            except AssertionError as e:
                return f"CTA {c}: {e}"
            continue
        live = [t for t, s in th.items() if s["st"] != "left"]
        if not live:
            continue
        c, t = rng.choice(live)
        s = th[c, t]
        n = s["n"]
        if s["st"] == "send":
            if n == H:
                s["st"] = "end"
                continue
            if not stopped(c, t):
                for side, count in ((0, role[t]["send"][0]), (1, role[t]["send"][1])):
                    if has(c, side):
                        flight += [(c - 1 if side == 0 else c + 1, 1 - side, n)] * count
            s["st"], s["side"] = "wait", 0
        elif s["st"] == "wait":
            if s["side"] == 2 or stopped(c, t):
                if s["side"] == 2 and not stopped(c, t):
                    for side, arms in ((0, t == 0), (1, t == TY - 1)):
                        if arms and has(c, side) and role[t]["recv"][side]:
                            sides[c][side].armed[n & 1] = n + 2
                meet((c, n), t, TY)
                s["st"] = "close"
                continue
            side = s["side"]
            if not (has(c, side) and role[t]["recv"][side]) or n in sides[c][side].done:
                s["side"] += 1
            elif rng.random() < limit:
                lost_at[c][t] = n
                meet((c, n), t, TY)
                s["st"] = "close"
        elif s["st"] == "close":
            if len(met[c, n]) == TY:
                if any(x == n for x in lost_at[c]):
                    lost[c] = True
                s["n"], s["st"] = n + 1, "send"
        elif s["st"] == "end":
            # What this thread waits for before it leaves: (side, hand-over).
            if protocol == "cta":
                meet("all", (c, t), C * TY)  # every CTA has sent what it sends
                first = min(x for x in lost_at[c] if x is not None) if lost[c] else None
                s["drain"] = [] if first is None else [(d, m) for m in (first + 1, first) for d in (0, 1)]
                s["st"] = "all"
            else:
                s["drain"] = [] if lost_at[c][t] is None else [(0, lost_at[c][t]), (1, lost_at[c][t])]
                s["st"] = "drain"
        elif s["st"] == "all":
            if len(met["all"]) == C * TY:
                s["st"] = "drain" if protocol == "cta" else "left"
        elif s["st"] == "drain":
            # Bounded, but far longer than bytes travel: it gives up on a phase only when nothing of it is on its way.
            if s["drain"]:
                d, m = s["drain"][-1]
                if not (has(c, d) and role[t]["recv"][d]) or m in sides[c][d].done or (c, d, m) not in flight:
                    s["drain"].pop()
                continue
            if protocol == "cta":
                s["st"] = "left"
            else:
                meet("all", (c, t), C * TY)
                s["st"] = "all"
        for q in range(C):
            gone[q] = gone[q] or all(th[q, u]["st"] == "left" for u in range(TY))
    return None


# (pairs per run, runs per column, halo rows): senders apart from receivers
# (120 x 90 mRNA/protein box), together, and mixed.
SHAPES = [(2, 4, 2), (3, 3, 1), (4, 2, 2), (1, 5, 1), (6, 1, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("C", [2, 3, 5])
def test_run_out_leaves_no_bytes_behind(shape, C):
    for seed in range(150):
        limit = (0.0, 0.02, 0.3, 1.0)[seed % 4]
        err = run(C, shape, 6, seed, "cta", limit)
        assert err is None, (seed, err)


def test_flag_per_thread_is_caught():
    """Threads that send and never receive go on sending after another thread's wait ran out."""
    fails = [run(3, (2, 4, 2), 6, seed, "thread", 0.3) for seed in range(150)]
    assert any(f and "not armed" in f for f in fails)
    fails = [run(3, (2, 4, 2), 2, seed, "thread", 1.0) for seed in range(150)]
    assert any(f and "has left" in f for f in fails)
