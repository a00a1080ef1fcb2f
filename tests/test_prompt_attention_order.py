"""The barriers between the softmax warps and the MMA warp of the tensor-core prompt attention, in every order in which the warps can run.

The barrier of P and how it is waited for are read from the source; the walk below runs the MMA warp (S(j), then P(j - 1) V(j - 1)) and three groups
of softmax warps through five tiles in every interleaving, with barriers that behave as mbarriers do (a phase ends with its last arrival, a
wait sees the parity of the phase).  No order may multiply a P that a group has not written, and none may get stuck."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_18911_b200", "csrc", "kg_prefill.cuh")
TILES, GROUPS = 5, 3


def walk(per_slot, parity):
    """per_slot: one barrier of P for each score tile in tensor memory, else one for all; parity(i): of the wait for tile i.  The first fault, or None."""
    arrivals = {"s0": 1, "s1": 1, "o0": 1, "o1": 1, "p0": GROUPS, "p1": GROUPS}
    names = sorted(arrivals)

    def arrive(bars, name):
        phase, pending = bars[names.index(name)]
        pending += 1
        new = (phase + 1, 0) if pending == arrivals[name] else (phase, pending)
        return tuple(new if n == name else b for n, b in zip(names, bars))

    def passed(bars, name, par):
        return bars[names.index(name)][0] & 1 != par

    def p(i):
        return f"p{i & 1 if per_slot else 0}"

    # the MMA warp's steps: S(0), S(1), PV(0), S(2), PV(1), ..., PV(TILES - 1)
    steps = [("S", 0)] + [x for j in range(1, TILES + 1) for x in ((("S", j),) if j < TILES else ()) + (("PV", j - 1),)]
    start = (0, (0,) * GROUPS, tuple((0, 0) for _ in names))
    seen, todo = {start}, [start]
    while todo:
        pc, soft, bars = todo.pop()
        nxt = []
        if pc < len(steps):
            kind, i = steps[pc]
            if kind == "S":
                if i < 2 or passed(bars, f"o{i & 1}", ((i >> 1) & 1) ^ 1):
                    nxt.append((pc + 1, soft, arrive(bars, f"s{i & 1}")))
            elif passed(bars, p(i), parity(i)):
                if min(soft) <= i:
                    return f"P({i}) is multiplied while the groups have written {soft} tiles"
                nxt.append((pc + 1, soft, arrive(bars, f"o{i & 1}")))
        for g, j in enumerate(soft):
            if j < TILES and passed(bars, f"s{j & 1}", (j >> 1) & 1) and (j < 2 or passed(bars, f"o{j & 1}", ((j - 2) >> 1) & 1)):
                nxt.append((pc, soft[:g] + (j + 1,) + soft[g + 1:], arrive(bars, p(j))))
        if not nxt and (pc < len(steps) or min(soft) < TILES):
            return f"stuck: the MMA warp before {steps[pc] if pc < len(steps) else 'its end'}, the groups have written {soft} tiles"
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


def test_no_order_of_the_warps_reads_p_early_or_gets_stuck():
    src = open(SRC).read()
    wait = re.search(r"gm_wait\(&?p_full(\[s\])?, \(unsigned\)(\(i >> 1\)|i) & 1u", src)
    arrive = re.search(r"mbar_arrive\(&?p_full(\[s\])?\)", src)
    assert wait and arrive and wait.group(1) == arrive.group(1)
    first, after = (int(re.search(rf"\*{n} = bar \+ (\d+)", src).group(1)) for n in ("p_full", "q_full"))
    per_slot = wait.group(1) is not None
    assert after - first == (2 if per_slot else 1)
    shift = 1 if ">>" in wait.group(2) else 0
    assert walk(per_slot, lambda i: (i >> shift) & 1) is None


def test_the_walk_sees_a_barrier_that_all_tiles_share():
    assert "is multiplied while" in walk(False, lambda i: i & 1) or "stuck" in walk(False, lambda i: i & 1)
