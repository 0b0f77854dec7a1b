"""Generated expansions of reduced loop nests, read on the CPU: the iterators of a
point are computed in arithmetic that may wrap, and looking for a nest's distinct
points costs little where there is nothing to find."""
import re
import time

import paper_2503_08946_gb300 as rc
from workloads.spec import Access, Array, GLOBAL, Loop, Model, Stmt, W, it, tid


def test_iterators_wrap():
    # values that fit 32 bits (64 bits) while the step times the point's number does not
    lo32, lo64 = -2_100_000_000, -(3 << 60)
    st = [Stmt([Access(0, W, ((it(0) // s + tid.x) % 97,))], loops=[Loop(lo, -lo, s), Loop(0, 2)])
          for lo, s in ((lo32, 1 << 21), (lo64, 1 << 52))]
    src = rc.rc_kernel_source(Model((2, 1, 1), (64, 1, 1), [Array("a", GLOBAL, (97,))], st))
    its = [e for e in re.findall(r"const (?:int|long long) i\d+ = (.*?);", src) if "*" in e]
    assert len(its) == 4 and all(re.search(r"\* \(unsigned(?: long long)?\)", e) for e in its), its
    assert not any(re.search(r"\* \((?:int|long long)\)", e) for e in its), its


def seconds(loops, index, n_stmts=400):
    st = [Stmt([Access(0, W, ((index + 3 * k + tid.x) % (1 << 20),))], loops=loops) for k in range(n_stmts)]
    m = Model((2, 1, 1), (64, 1, 1), [Array("a", GLOBAL, (1 << 20,))], st)
    times = []
    for _ in range(3):
        t = time.perf_counter()
        src = rc.rc_kernel_source(m)
        times.append(time.perf_counter() - t)
    return min(times), src


def test_distinct_nests_cost_little():
    # (lower bounds that move with an outer iterator: no points are compared)
    ref, src = seconds([Loop(0, 64), Loop(it(0), it(0) + 64)], 64 * it(0) + it(1))
    assert "pts0[" not in src
    for loops, index in (([Loop(0, 64), Loop(0, 64)], 64 * it(0) + it(1)),
                         ([Loop(0, 16), Loop(0, 16), Loop(0, 16)], it(0) + 16 * it(2) + 256 * it(1)),
                         ([Loop(0, 64), Loop(0, 64)], 63 * it(0) + it(1) + (it(1) // 7) * 64)):
        t, src = seconds(loops, index)
        assert "pts0[" not in src
        assert t < 3 * ref, (t, ref)
    # nests that are reduced until constant memory is full
    t, src = seconds([Loop(0, 64), Loop(0, 64)], 31 * it(0) + it(1))
    assert "pts0[" in src and "pts399[" not in src
    assert t < 3 * ref, (t, ref)
