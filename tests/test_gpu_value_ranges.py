"""Generated expansions in 32-bit arithmetic: rows whose values lie at the edges of
32 bits (and of 64), negative dividends, divisors beyond 32 bits, table values,
loops that run up to the edge, checks that the ranges decide; and accesses that
repeat their instance in the innermost loop.  Against the oracle."""
import pytest

import oracle
from workloads.rng import SplitMix64
from workloads.spec import A, Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, bid, const, it, load, tid

pytestmark = pytest.mark.gpu
B31, B32, B62 = 1 << 31, 1 << 32, 1 << 62


@pytest.fixture(scope="module")
def rc():
    import torch
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


@pytest.fixture(autouse=True)
def jit_on(monkeypatch):
    monkeypatch.setenv("RC_JIT", "1")


def check(rc, m, opts=None):
    h = rc.rc_model_create(m)
    assert rc.rc_model_layout(h)["expand_jit"] == 1
    got, exp = rc.check(h, opts), oracle.check(m)
    assert (got.status, got.instances) == (exp.status, exp.instances), (m.name, got, exp)
    if exp.status:
        assert (got.oob_stmt, got.oob_access, got.oob_gtid, got.oob_dim) == \
            (exp.oob_stmt, exp.oob_access, exp.oob_gtid, exp.oob_dim), m.name
    else:
        assert (got.verdict, got.racy_cells, got.witness) == (exp.verdict, exp.racy_cells, exp.witness), m.name


def one(exprs, loops=(), guards=(), tables=(), ext=97, phase=const(0), n_phases=1, block=33):
    a = Array("a", GLOBAL, (ext,))
    acc = [Access(0, W, (e % ext,)) for e in exprs]
    return Model((3, 1, 1), (block, 1, 1), [a], [Stmt(acc, loops=list(loops), guards=list(guards), phase=phase)],
                 n_phases=n_phases, tables=[list(t) for t in tables], name="r")


EDGE = [B31 - 1, B31, -B31, -B31 - 1, B31 - 33, -B31 + 65, B32, -B32 - 5, B62 - 100, -B62 + 100]


@pytest.mark.parametrize("c0", EDGE)
@pytest.mark.parametrize("d", [1, 3, 7, 32, 1000003, B31 - 1, B31, B32 + 1])
def test_terms_at_the_edge(rc, c0, d):
    x = const(c0) + tid.x - 16 * bid.x
    check(rc, one([x // d, x % d, (x // d) * 5 + x % d, (x % d) // 3]))


@pytest.mark.parametrize("c0", EDGE)
def test_coefficients_beyond_32_bits(rc, c0):
    check(rc, one([c0 * tid.x + (1 - c0) * tid.x, (c0 * bid.x) // 64 + tid.x, const(c0) + tid.x]))


@pytest.mark.parametrize("c0", EDGE[:8])
def test_loops_at_the_edge(rc, c0):
    check(rc, one([it(0) + tid.x, it(0) // 5], loops=[Loop(const(c0), const(c0 + 7), 3)]))
    check(rc, one([it(0) * 3 + it(1)], loops=[Loop(const(c0) + tid.x, const(c0 + 9), 2), Loop(it(0) - c0, const(6))]))


@pytest.mark.parametrize("v", [0, 5, B31 - 1, B31, -B31 - 1, B62])
def test_table_values(rc, v):
    t = [3, v, -2, v - 1]
    check(rc, one([load(0, tid.x % 6), load(0, load(0, tid.x % 4) % 5) // 7], tables=[t]))
    check(rc, one([it(0) + tid.x], loops=[Loop(load(0, tid.x % 2) - load(0, tid.x % 2), load(0, const(0)))], tables=[t]))


@pytest.mark.parametrize("shift", [-1, 0, 1, 2])
def test_decided_and_undecided_bounds(rc, shift):
    # in bounds for every thread, or out of bounds at one end; a phase that leaves its range
    a, b = Array("a", GLOBAL, (99, 5)), Array("b", SHARED, (33,))
    st = [Stmt([Access(0, W, (33 * bid.x + tid.x + shift - 1, it(0))), Access(1, R, (tid.x,))], loops=[Loop(0, 5)]),
          Stmt([Access(1, W, (tid.x,))], phase=it(0), loops=[Loop(0, 2 + (shift > 1))], guards=[32 - tid.x])]
    check(rc, Model((3, 1, 1), (33, 1, 1), [a, b], st, n_phases=2, name=f"b{shift}"))


@pytest.mark.parametrize("seed", range(24))
def test_repeated_accesses(rc, seed):
    """Accesses fixed in the innermost loop beside ones that move, in nests of
    constant and of thread-dependent trips, with guards and intervals that move."""
    rng = SplitMix64(0x4E9 ^ seed * 0x9E3779B97F4A7C15)
    s, g = Array("s", SHARED, (40,)), Array("g", GLOBAL, (300,))
    st = []
    for _ in range(4):
        n = rng.uniform_int(1, 3)
        loops = [Loop(rng.below(2), const(rng.uniform_int(1, 4)) if rng.chance(0.4) else tid.x % 4 + 1) for _ in range(n)]
        acc = []
        for _ in range(rng.uniform_int(1, 4)):
            e = rng.uniform_int(0, 3) * tid.x + rng.uniform_int(0, 2) * bid.x + rng.below(9)
            for l in range(n):
                if rng.chance(0.35):
                    e = e + rng.uniform_int(1, 3) * it(l)
            acc.append(Access(0, (R, W, A)[rng.below(3)], (e % 40,)) if rng.chance(0.5) else
                       Access(1, (R, W, A)[rng.below(3)], (e % 300,)))
        guards = [rng.below(20) - tid.x + it(n - 1)] if rng.chance(0.5) else []
        ph = const(rng.below(3))
        st.append(Stmt(acc, loops=loops, guards=guards, phase=ph))
    m = Model((3, 1, 1), (37, 1, 1), [s, g], st, n_phases=3, name=f"rep{seed}")
    check(rc, m)
    check(rc, m, {"flags": 8})
