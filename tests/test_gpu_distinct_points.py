"""Generated expansions of statements whose loop nests repeat their instances: the
check makes a key per distinct point and counts every point; rc_expand_keys
writes all of them.  Against the oracle, generated kernels forced."""
import numpy as np
import pytest

import oracle
import workloads as w
from tests.test_gpu_parity import decode_keys, keyed_rows
from workloads.spec import Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, A, bid, const, it, load, tid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


@pytest.fixture
def jit_on(monkeypatch):
    monkeypatch.setenv("RC_JIT", "1")


def model(case):
    sh, gl = Array("s", SHARED, (48,)), Array("g", GLOBAL, (4000,))
    i, j, k = it(0), it(1), it(2)
    loops = [Loop(0, 5), Loop(2, 14, 3), Loop(const(-1), const(3))]
    stmts = {
        # invariant in every loop, in one loop, moving along two loops, with a term
        "invariant": [Stmt([Access(0, W, (tid.x % 48,))], loops=loops)],
        "one_loop": [Stmt([Access(1, W, (tid.x * 4 + i,)), Access(0, R, ((tid.x + i) % 48,))], loops=loops)],
        "diagonal": [Stmt([Access(1, W, ((tid.x * 3 + i - j + 2 * k) % 4000,))], loops=loops)],
        "term": [Stmt([Access(1, W, (((tid.x + 2 * i + 4 * j) // 3) % 4000,)), Access(0, A, (tid.x % 7,))], loops=loops)],
        # guards and intervals that move with the loops, or do not
        "guard_moves": [Stmt([Access(0, W, (tid.x % 48,))], loops=loops, guards=[i + j - 6], phase=const(0)),
                        Stmt([Access(0, R, ((tid.x + 1) % 48,))], phase=const(1))],
        "guard_stays": [Stmt([Access(0, W, ((tid.x + j) % 48,))], loops=loops, guards=[tid.x - 5]),
                        Stmt([Access(0, R, ((tid.x + 1) % 48,))], loops=[Loop(0, 9)])],
        "phase_moves": [Stmt([Access(0, W, (tid.x % 48,))], loops=loops, phase=i)],
        # bounds that move with the thread (distinct) or with an outer iterator (all points kept)
        "thread_bound": [Stmt([Access(1, W, (i + 2 * j,))], loops=[Loop(tid.x, tid.x + 6), Loop(0, 4)])],
        "outer_bound": [Stmt([Access(1, W, (i + j,))], loops=[Loop(0, 6), Loop(i, i + 4)])],
        # a nest without keys beside one with them, and a nest of thread-dependent trips
        "mixed": [Stmt([Access(1, R, (tid.x + i,))], loops=loops), Stmt([Access(0, W, (tid.x % 48,))], loops=[Loop(0, 7)]),
                  Stmt([Access(0, W, ((tid.x + i) % 48,))], loops=[Loop(0, tid.x % 3)])],
        "out_of_bounds": [Stmt([Access(0, W, (tid.x + i,))], loops=[Loop(0, 3), Loop(0, 5)])],
        "table": [Stmt([Access(0, W, (load(0, i) % 48,))], loops=[Loop(0, 4), Loop(0, 3)])],
    }[case]
    return Model((3, 1, 1), (50, 1, 1), [sh, gl], stmts, n_phases=5, name=case, tables=[[3, 1, 4, 1]])


CASES = ["invariant", "one_loop", "diagonal", "term", "guard_moves", "guard_stays", "phase_moves", "thread_bound",
         "outer_bound", "mixed", "out_of_bounds", "table"]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("flags", [0, 8])      # bucket path, radix sort
def test_check(rc, jit_on, case, flags):
    m = model(case)
    got, exp = rc.check(m, {"flags": flags}), oracle.check(m)
    assert (got.status, got.instances) == (exp.status, exp.instances)
    if exp.status == 0:
        assert (got.verdict, got.racy_cells, got.witness) == (exp.verdict, exp.racy_cells, exp.witness)
    else:
        assert (got.oob_stmt, got.oob_access, got.oob_gtid, got.oob_dim) == \
            (exp.oob_stmt, exp.oob_access, exp.oob_gtid, exp.oob_dim)


@pytest.mark.parametrize("case", ["diagonal", "mixed", "guard_moves"])
def test_expand_keys_writes_every_point(rc, jit_on, case):
    m = model(case)
    h = rc.rc_model_create(m)
    lay = rc.rc_model_layout(h)
    keys = torch.empty(lay["key_slots"], dtype=torch.int64, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    rc.rc_expand_keys(h, rc.workspace(rc.rc_workspace_size(h)), keys, cnt)
    torch.cuda.synchronize()
    exp = oracle.expand(m)
    assert int(cnt.item()) == len(exp)
    assert np.array_equal(decode_keys(keys.cpu().numpy().view(np.uint64), lay, m), keyed_rows(exp, m))


@pytest.mark.parametrize("case", ["diagonal", "guard_moves", "mixed"])
def test_wide(rc, jit_on, case):
    m = model(case)
    m.arrays[1] = Array("g", GLOBAL, (4000, 1 << 44))
    for s in m.stmts:
        s.accesses[:] = [Access(a.array, a.kind, a.index + (const(1 << 43),)) if a.array == 1 else a for a in s.accesses]
    assert rc.rc_model_layout(rc.rc_model_create(m))["wide"] == 1
    got, exp = rc.check(m), oracle.check(m)
    assert (got.status, got.instances, got.racy_cells, got.witness) == (exp.status, exp.instances, exp.racy_cells, exp.witness)
