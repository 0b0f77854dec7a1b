"""Generated expansions of reduced loop nests, read on the CPU: the iterators of a
point are computed in arithmetic that may wrap."""
import re

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
