"""Barrier protocol of the bf16 many-nets kernel (csrc/tc_kernels.cu), every
interleaving on the CPU.  A parity wait sees one phase back: where a barrier
can complete twice before its waiter has looked, the waiter blocks on a phase
that needs the waiter itself.  The model has the forward warp, the gradient
warp, two threads of each epilogue group (for its 256) and commits that arrive
any time after their issue, in order; the barriers of the hand-overs between
MMAs and epilogue are indexed as the source's constants say."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1908_07847_gb300", "csrc", "tc_kernels.cu")


def program(T, E, nz1f, ndf):
    """Programs of the six roles over T tiles and E epochs, and the arrivals a
    barrier takes: ('w', bar, n) waits for completion n of bar, ('a', bar)
    arrives, ('c', q, bar) commits to MMA queue q.  Half tile s = 2 tile + group."""
    w0, w1, epi = [], [], [[], []]

    def use(name, s, n):
        return (name, s % n), s // n + 1

    for it in range(T * E):
        t, e = it % T, it // T
        if t == 0 and e > 0:
            w0.append(("w", ("W",), e))
        for g in range(2):
            s = 2 * it + g
            if s >= 3:                                # the buffer's previous d1 has been read
                w0.append(("w", *use("GD", s - 3, 3)))
            w0.append(("c", 0, use("Z1F", s, nz1f)[0]))
            w1 += [("w", *use("DF", s, ndf)), ("c", 1, use("GD", s, 3)[0])]
            epi[g] += [("w", *use("Z1F", s, nz1f)), ("a", ("EPI", g)), ("w", ("EPI", g), it + 1),
                       ("a", use("DF", s, ndf)[0])]
        if t == T - 1:
            w1.append(("c", 1, ("EPOCH",)))
            for p in epi:
                p += [("w", ("EPOCH",), e + 1), ("a", ("EPIA",)), ("w", ("EPIA",), e + 1), ("a", ("W",))]
    count = {"W": 4, "EPIA": 4, "EPI": 2, "DF": 2}
    return [w0, w1, epi[0], epi[0], epi[1], epi[1]], count


def explore(T, E, nz1f, ndf):
    """None, or what goes wrong first in some interleaving."""
    progs, count = program(T, E, nz1f, ndf)
    bars = sorted({o[2] if o[0] == "c" else o[1] for p in progs for o in p})
    idx = {b: i for i, b in enumerate(bars)}
    start = ((0,) * 6, (0,) * len(bars), ((), ()))    # positions, arrivals so far, commits in flight
    seen, stack = {start}, [start]
    while stack:
        pos, arr, qs = stack.pop()

        def arrived(b):
            return tuple(v + (i == idx[b]) for i, v in enumerate(arr))

        nxt = [(pos, arrived(qs[q][0]), tuple(x[1:] if i == q else x for i, x in enumerate(qs)))
               for q in range(2) if qs[q]]
        for i, p in enumerate(progs):
            if pos[i] == len(p):
                continue
            o, a, n = p[pos[i]], arr, qs
            if o[0] == "w":
                done = arr[idx[o[1]]] // count.get(o[1][0], 1)
                passes = (done ^ o[2]) & 1 == 0       # the last completed phase has the parity waited for
                if passes != (done >= o[2]):
                    return "role %d, completion %d of %s: %d done" % (i, o[2], o[1], done)
                if not passes:
                    continue
            elif o[0] == "a":
                a = arrived(o[1])
            else:
                n = tuple(x + (o[2],) if j == o[1] else x for j, x in enumerate(qs))
            nxt.append((tuple(v + (j == i) for j, v in enumerate(pos)), a, n))
        if not nxt and any(pos[i] < len(p) for i, p in enumerate(progs)):
            return "deadlock at %s" % (pos,)
        for s in nxt:
            if s not in seen:
                seen.add(s)
                stack.append(s)
    return None


@pytest.mark.parametrize("T,E", [(1, 3), (2, 2), (3, 2), (5, 1)])
def test_no_wait_of_the_kernel_misses_a_phase(T, E):
    src = open(SRC).read()
    nz1 = int(re.search(r"constexpr int NZ1 = (\d+);", src).group(1))
    nz1f = int(re.search(r"constexpr int NZ1F = (\d+) \* NZ1;", src).group(1)) * nz1
    ndf = {"NZ1": nz1}[re.search(r"constexpr int NDF = (\w+);", src).group(1)]
    assert nz1 == 3 and explore(T, E, nz1f, ndf) is None


def test_one_barrier_a_group_misses_phases():
    assert explore(2, 2, 2, 3) is not None and explore(2, 2, 6, 2) is not None
