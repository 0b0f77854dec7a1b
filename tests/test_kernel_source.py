"""The generated expansion's tables fit constant memory whatever the number of
statements, and hold every point of a nest once."""
import re

import pytest

import paper_2503_08946_gb300 as rc
from workloads.spec import Access, Array, GLOBAL, Loop, Model, Stmt, W, it, tid


def constant_bytes(src):
    n = 0
    for t, k in re.findall(r"__constant__ (ushort2|uint3) \w+\[(\d+)\]", src):
        n += int(k) * {"ushort2": 4, "uint3": 12}[t]
    return n


@pytest.mark.parametrize("n_stmts", [1, 36, 400, 1100, 4096])
def test_constant_tables_fit(n_stmts):
    a = Array("a", GLOBAL, (4096,))
    st = [Stmt([Access(0, W, ((tid.x + it(0) + it(1) + k) % 4096,))], loops=[Loop(0, 40), Loop(0, 40)]) for k in range(n_stmts)]
    src = rc.rc_kernel_source(Model((2, 1, 1), (64, 1, 1), [a], st))
    assert 0 < constant_bytes(src) <= 64 << 10
    # i + j takes 79 values over 40 x 40 points
    tabs = re.findall(r"pts\d+\[(\d+)\] = \{(.*?)\};", src)
    assert tabs and all(int(n) == 79 for n, _ in tabs)
    for _, body in tabs[:3]:
        pairs = [tuple(map(int, p)) for p in re.findall(r"\{(\d+),(\d+)\}", body)]
        assert sum(times for _, times in pairs) == 1600 and len({p for p, _ in pairs}) == 79
