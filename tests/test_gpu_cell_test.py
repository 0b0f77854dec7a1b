"""The cell test in shared memory (bucket path without a sort): models without
atomics and scopes against the oracle at the edges of its buckets -- one key, the
unpartitioned bucket, one and two partition passes, buckets above the register
capacity (hot cells), candidate cells in several windows of the table, sixteen
intervals, and the largest key word below the cell."""
import pytest

import oracle
import workloads as w
from workloads.rng import SplitMix64
from workloads.spec import A, Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, bid, const, it, load, tid

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import torch
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


def check(rc, model, opts=None):
    got, exp = rc.check(model, opts), oracle.check(model)
    assert (got.status, got.instances) == (exp.status, exp.instances) == (0, exp.instances), (model.name, got, exp)
    assert (got.verdict, got.racy_cells, got.witness) == (exp.verdict, exp.racy_cells, exp.witness), (model.name, got, exp)


def shared_mix(blocks, threads, cells, phases, scope=SHARED, hot=1):
    """Cells written by one thread in several intervals and read by another one in
    intervals with and without a write: the candidates of the test's third step,
    about a third of them racy."""
    a = Array("a", scope, (cells,))
    own, other = tid.x % cells, (tid.x * 7 + 3) % cells
    stmts = [Stmt([Access(0, W, (own,))], phase=const(p), loops=[Loop(0, hot)], name=f"w{p}")
             for p in range(0, phases, 2)]
    stmts += [Stmt([Access(0, R, (other,))], phase=const(p), guards=[tid.x % 3 - (1 if p % 2 == 0 else 0)],
                   loops=[Loop(0, hot)], name=f"r{p}") for p in range(phases)]
    return Model((blocks, 1, 1), (threads, 1, 1), [a], stmts, n_phases=phases, name=f"mix_{blocks}_{threads}_{cells}_{phases}")


@pytest.mark.parametrize("phases", [1, 2, 7, 16])
@pytest.mark.parametrize("blocks,threads", [(1, 1), (1, 33), (3, 96), (64, 256)])
def test_candidates(rc, blocks, threads, phases):
    check(rc, shared_mix(blocks, threads, max(1, threads), phases))
    check(rc, shared_mix(blocks, threads, max(1, threads // 3), phases, scope=GLOBAL))


def test_many_candidates_of_sixteen_intervals(rc):
    # ~500 candidate cells and more per bucket: several windows of the table
    check(rc, shared_mix(40, 512, 512, 16))


@pytest.mark.parametrize("cells", [1, 3, 40])
def test_hot_cells_exceed_the_registers(rc, cells):
    # tens of thousands of keys in a few cells: a bucket read again in every step
    check(rc, shared_mix(30, 200, cells, 4, hot=9))
    check(rc, shared_mix(30, 200, cells, 1, scope=GLOBAL, hot=9))


def word_model(block_extra):
    """Interval, block, thread and kind fill exactly (or just exceed) 32 bits;
    a few threads are left by the guards."""
    blocks, threads = 1 << 17, 512        # 17 + 9 bits, kind 1, intervals 4 (32 phases would leave the path) + 1
    a = Array("a", GLOBAL, (1 << (5 + block_extra),))
    i = (tid.x + bid.x) % (1 << (5 + block_extra))
    g = [const(3) - tid.x, const(40) - bid.x]
    return Model((blocks << block_extra, 1, 1), (threads, 1, 1), [a],
                 [Stmt([Access(0, W, (i,))], phase=const(15), guards=g),
                  Stmt([Access(0, R, ((i + 1) % (1 << (5 + block_extra)),))], phase=const(0), guards=g)], n_phases=16,
                 name=f"word{block_extra}")


@pytest.mark.parametrize("extra", [0, 1])
def test_key_word_widths(rc, extra):
    m = word_model(extra)
    h = rc.rc_model_create(m)
    assert rc.rc_model_layout(h)["cell_shift"] == 31 + extra
    check(rc, m)


@pytest.mark.parametrize("n", [1, 31, 4320, 4321, 4700, 4701, 5120, 5121])
def test_bucket_edges(rc, n):
    a = Array("a", GLOBAL, (max(1, n // 2),))
    m = Model((1, 1, 1), (1, 1, 1), [a], [Stmt([Access(0, W, (it(0) % max(1, n // 2),))], loops=[Loop(0, n)])])
    check(rc, m)
    m2 = Model((2, 1, 1), (1, 1, 1), [a], m.stmts)
    check(rc, m2)


@pytest.mark.parametrize("parts", [2, 16])
def test_hash_parts_report_the_smallest_cell(rc, parts):
    m = shared_mix(24, 128, 128, 5)
    whole = rc.check(m)
    got = [rc.check(m, {"part_count": parts, "part_index": i}) for i in range(parts)]
    assert sum(r.racy_cells for r in got) == whole.racy_cells
    assert min(r.witness for r in got if r.verdict) == whole.witness


def atomic_mix(seed, blocks, threads, cells, phases, scope):
    """Reads, writes and atomics of few cells in few (or many) intervals, each
    statement by a part of the threads and blocks: every combination of kinds in
    a cell, an interval and a block turns up over the seeds."""
    rng = SplitMix64(0xA70 ^ seed * 0x9E3779B97F4A7C15)
    a = Array("a", scope, (cells,))
    stmts = []
    for s in range(rng.uniform_int(2, 9)):
        kind = (R, A, A, W)[rng.below(4)]
        i = (rng.uniform_int(0, 3) * tid.x + rng.uniform_int(0, 2) * bid.x + rng.below(cells)) % cells
        guards = [rng.below(threads) - tid.x] if rng.chance(0.5) else [rng.uniform_int(0, 2) - tid.x % 3]
        if rng.chance(0.3):
            guards.append(const(0) - bid.x % 2)
        stmts.append(Stmt([Access(0, kind, (i,))], phase=const(rng.below(phases)), guards=guards, name=f"{kind}{s}"))
    return Model((blocks, 1, 1), (threads, 1, 1), [a], stmts, n_phases=phases, name=f"amix{seed}")


@pytest.mark.parametrize("seed", range(60))
def test_atomics(rc, seed):
    scope = (SHARED, GLOBAL)[seed & 1]
    check(rc, atomic_mix(seed, 1 + seed % 3, 40, 1 + seed % 13, 1 + seed % 5, scope))
    check(rc, atomic_mix(seed, 3, 64, 64 if scope == SHARED else 700, 16, scope))


@pytest.mark.parametrize("seed", range(8))
def test_atomics_partitioned(rc, seed):
    check(rc, atomic_mix(100 + seed, 60, 256, 200, 1 + seed, (SHARED, GLOBAL)[seed & 1]))


@pytest.mark.parametrize("phases", [17, 32, 33, 64, 65])
def test_many_intervals(rc, phases):
    m = shared_mix(20, 192, 100, phases)          # 65,280 key slots and more at 17 intervals and more
    n = rc.rc_model_layout(rc.rc_model_create(m))["key_slots"]
    assert n >= 65536 or phases == 17
    check(rc, m)
    check(rc, atomic_mix(7, 300, 256, 50, phases, SHARED))
    check(rc, atomic_mix(8, 300, 256, 3000, phases, GLOBAL))


# ---- hashed tables (cell spaces too sparse for a slot per cell) ----

@pytest.mark.parametrize("row_bits", [8, 16, 20, 24])
@pytest.mark.parametrize("blocks", [1, 9, 64])
def test_sparse_rows(rc, row_bits, blocks):
    check(rc, w.random_affine(11 + row_bits, n_blocks=blocks, block=64, n_stmts=20, plant=True,
                              row_global=1 << row_bits))


def same_bucket(n, atomic=False, cb=24):
    """n cells that share the top hash bits (hash values 0 .. n - 1), so that they
    lie in one bucket: more written cells than its table has slots.  Thread t
    writes cell t; every third cell is read by the next thread, every fifth in
    the same interval."""
    inv = pow(0x9E3779B97F4A7C15, -1, 1 << 64)
    cells = [(h * inv) % (1 << cb) for h in range(n)]
    cells = [c if c < (1 << cb) - 1 else 0 for c in cells]
    a = Array("a", GLOBAL, ((1 << cb) - 1,))
    block = 250
    g = bid.x * block + tid.x
    kind = A if atomic else W
    stmts = [Stmt([Access(0, kind, (load(0, g),))], phase=const(0)),
             Stmt([Access(0, R, (load(0, (g + 1) % n),))], phase=const(1), guards=[const(0) - g % 3]),
             Stmt([Access(0, R, (load(0, (g + 7) % n),))], phase=const(0), guards=[const(0) - g % 5, const(100) - bid.x])]
    return Model((n // block, 1, 1), (block, 1, 1), [a], stmts, n_phases=2, tables=[cells], name=f"same_bucket{n}")


@pytest.mark.parametrize("atomic", [False, True])
@pytest.mark.parametrize("n", [250, 1500, 8000, 20000, 40000])
def test_more_written_cells_than_slots(rc, n, atomic):
    check(rc, same_bucket(n, atomic))


@pytest.mark.parametrize("seed", range(6))
def test_sparse_atomics_and_batches(rc, seed):
    rng = SplitMix64(seed)
    big = Array("a", GLOBAL, (5000, 1 << 17))
    ms = []
    for k in range(7):
        i = (rng.uniform_int(1, 4) * tid.x + rng.uniform_int(0, 9) * bid.x) % 5000
        st = [Stmt([Access(0, (R, W, A)[rng.below(3)], (i + const(j % 2), const((1 << 16) + 3 * j)))],
                   phase=const(rng.below(3))) for j in range(4)]
        ms.append(Model((1 + rng.below(40), 1, 1), (32 * (1 + rng.below(4)), 1, 1), [big], st, n_phases=3, name=f"sp{k}"))
    exp = [oracle.check(m) for m in ms]
    for m, e in zip(ms, exp):
        got = rc.check(m)
        assert (got.status, got.racy_cells, got.witness) == (e.status, e.racy_cells, e.witness), m.name
    h = [rc.rc_model_create(m) for m in ms]
    got = rc.rc_report(rc.rc_check_batch(h, None, rc.workspace(rc.rc_batch_workspace_size(h, None))))
    assert [(g.status, g.instances, g.racy_cells, g.witness) for g in got] == \
        [(e.status, e.instances, e.racy_cells, e.witness) for e in exp]
