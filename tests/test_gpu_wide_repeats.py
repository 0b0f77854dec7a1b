"""Wide models (checked in cell-range chunks) whose accesses stay in a cell while the
innermost loop runs and whose interval moves with an outer one: the generated count
and route kernel keeps a key per interval.  Against the oracle."""
import pytest

import oracle
import workloads as w
from workloads.rng import SplitMix64
from workloads.spec import A, Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, bid, const, it, tid

pytestmark = pytest.mark.gpu
FAR = 1 << 44


@pytest.fixture(scope="module")
def rc():
    import torch
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


def check(rc, monkeypatch, m, racy=None):
    exp = oracle.check(m)
    assert exp.status == 0 and (racy is None or exp.racy_cells == racy)
    for jit in "10":
        monkeypatch.setenv("RC_JIT", jit)
        h = rc.rc_model_create(m)
        assert rc.rc_model_layout(h)["wide"] == 1
        got = rc.check(h)
        assert (got.status, got.instances, got.verdict, got.racy_cells, got.witness) == \
            (exp.status, exp.instances, exp.verdict, exp.racy_cells, exp.witness), (m.name, jit)


# thread-dependent trips; constant trips with an access that makes the points
# distinct; a lower bound that moves with the outer iterator
INNER = {"thread": Loop(0, tid.x % 3 + 1), "moving": Loop(0, 5), "outer": Loop(it(0), it(0) + 2)}


@pytest.mark.parametrize("inner", sorted(INNER))
@pytest.mark.parametrize("scope", [SHARED, GLOBAL])
def test_interval_of_an_outer_loop(rc, monkeypatch, inner, scope):
    arrays = [Array("g", GLOBAL, (4000, FAR)), Array("s", scope, (64,))]
    st = [Stmt([Access(1, W, (tid.x,)), Access(0, W, ((bid.x * 50 + tid.x) * 5 + it(1) % 5, const(FAR // 2)))],
               loops=[Loop(0, 3), INNER[inner]], phase=it(0)),
          Stmt([Access(1, R, ((tid.x + 1) % 64,))], phase=const(1))]
    # in each block cells 1..49 are written by their own thread and read by the one before
    check(rc, monkeypatch, Model((3, 1, 1), (50, 1, 1), arrays, st, n_phases=3, name=inner),
          racy=147 if scope == SHARED else 50)


def test_last_interval_of_a_wide_cell(rc, monkeypatch):
    g = Array("g", GLOBAL, (4000, 1 << 46))
    st = [Stmt([Access(0, W, (tid.x, const(7)))], loops=[Loop(0, 3), Loop(0, tid.x % 3 + 1)], phase=it(0)),
          Stmt([Access(0, R, ((tid.x + 1) % 50, const(7)))], phase=const(2))]
    check(rc, monkeypatch, Model((1, 1, 1), (50, 1, 1), [g], st, n_phases=3), racy=50)


@pytest.mark.parametrize("trailing", [True, False])
def test_ge_spmm(rc, monkeypatch, trailing):
    m = w.ge_spmm_csr([70, 0, 33, 1, 96, 40, 32, 5], N=64, K=2, trailing_barrier=trailing)
    m.arrays[4] = Array("C", GLOBAL, (8, 64, FAR))
    for s in m.stmts:
        s.accesses[:] = [Access(a.array, a.kind, a.index + (const(FAR - 1),)) if a.array == 4 else a for a in s.accesses]
    check(rc, monkeypatch, m, racy=0 if trailing else 2 * 2 * (32 + 1 + 32 + 8))


@pytest.mark.parametrize("seed", range(24))
def test_random(rc, monkeypatch, seed):
    rng = SplitMix64(0x71DE ^ seed * 0x9E3779B97F4A7C15)
    s, g = Array("s", SHARED, (40,)), Array("g", GLOBAL, (300, FAR))
    st = []
    for _ in range(5):
        n = rng.uniform_int(1, 3)
        loops = [Loop(rng.below(2), const(rng.uniform_int(2, 4)) if l == 0 or rng.chance(0.4) else tid.x % 4 + 1)
                 for l in range(n)]
        acc = []
        for _ in range(rng.uniform_int(1, 3)):
            e = rng.uniform_int(1, 3) * tid.x + rng.uniform_int(0, 2) * bid.x + rng.below(9)
            for l in range(n):
                if rng.chance(0.3):
                    e = e + rng.uniform_int(1, 3) * it(l)
            kind = (R, R, W, A)[rng.below(4)]
            acc.append(Access(0, kind, (e % 40,)) if rng.chance(0.7) else
                       Access(1, kind, (e % 300, const(FAR - 3) - it(0))))
        guards = [rng.below(20) - tid.x + it(n - 1)] if rng.chance(0.4) else []
        st.append(Stmt(acc, loops=loops, guards=guards, phase=it(0) + rng.below(3) if rng.chance(0.7) else const(1)))
    check(rc, monkeypatch, Model((3, 1, 1), (37, 1, 1), [s, g], st, n_phases=6, name=f"wr{seed}"))
