"""Cells that are written in several intervals and read by other threads (every one
a candidate of the cell test's third step): several tables of candidates, threads of
up to 15 bits and more, buckets in registers and larger ones, against the oracle; and
correct tile buffers on the default path against the radix path: the same result, in
no more time.  The line of 1.25 is the spread of single timings; both are medians of
the same process."""
import statistics
import time

import pytest

import oracle
from workloads.spec import A, Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, bid, const, it, tid

pytestmark = pytest.mark.gpu
LSD = 8


@pytest.fixture(scope="module")
def rc():
    import torch
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


def tiles(log_threads, phases, block=256):
    """written in even intervals by its owner, read by the neighbour in odd ones"""
    t = Array("t", SHARED, (block,))
    return Model(((1 << log_threads) // block, 1, 1), (block, 1, 1), [t],
                 [Stmt([Access(0, W, (tid.x,))], loops=[Loop(0, phases, 2)], phase=it(0)),
                  Stmt([Access(0, R, ((tid.x + 1) % block,))], loops=[Loop(1, phases, 2)], phase=it(0))],
                 n_phases=phases, name=f"tiles{log_threads}_{phases}")


def compare(rc, m, verdict):
    h = rc.rc_model_create(m)
    seen, us = [], []
    for flags in (0, LSD):
        opts = {"flags": flags}
        ws = rc.workspace(rc.rc_workspace_size(h, opts))
        t = []
        for k in range(9):
            t0 = time.perf_counter()
            r = rc.rc_report(rc.rc_check(h, opts, ws))[0]
            t.append(time.perf_counter() - t0)
        del ws
        seen.append((r.status, r.verdict, r.racy_cells, r.instances, r.witness))
        us.append(1e6 * statistics.median(t[2:]))
    assert seen[0] == seen[1] and seen[0][:3] == (0, verdict, verdict), (m.name, seen)
    assert us[0] < 1.25 * us[1], (m.name, us)


@pytest.mark.parametrize("log_threads,phases", [(18, 40), (20, 16), (20, 17), (20, 40), (20, 64), (21, 32), (22, 16), (23, 8)])
def test_tile_buffers(rc, log_threads, phases):
    compare(rc, tiles(log_threads, phases), 0)


def crowd(blocks, block, phases, kind, hot=0, racy=True):
    """a cell per thread, changed by its owner in two intervals and read by the
    neighbour between and after them; every 37th one is read where it is changed;
    `hot` global cells that all threads only add to (or, written, race)"""
    a, h = Array("a", SHARED, (block,)), Array("h", GLOBAL, (max(1, hot),))
    own, nxt = (tid.x,), ((tid.x + 1) % block,)
    p, q = phases // 3, phases - 2
    st = [Stmt([Access(0, kind, own)], phase=const(x)) for x in (p, q)]
    st += [Stmt([Access(0, R, nxt)], phase=const(x)) for x in ((p + q) // 2, phases - 1) if x not in (p, q)]
    if racy:
        st.append(Stmt([Access(0, R, nxt)], phase=const(q), guards=[const(0) - tid.x % 37]))
    if hot:
        st.append(Stmt([Access(1, kind, (tid.x % hot,))], phase=const(0)))
    return Model((blocks, 1, 1), (block, 1, 1), [a, h], st, n_phases=phases, name=f"crowd{blocks}_{block}_{phases}{kind}{hot}")


def against_oracle(rc, m):
    got, exp = rc.check(m), oracle.check(m)
    assert (got.status, got.instances, got.verdict, got.racy_cells, got.witness) == \
        (0, exp.instances, exp.verdict, exp.racy_cells, exp.witness), (m.name, got, exp)


@pytest.mark.parametrize("kind", [W, A])
@pytest.mark.parametrize("phases", [4, 16, 33, 64])
@pytest.mark.parametrize("blocks,block", [(400, 256), (101, 1000), (3, 32768), (3, 32769), (2, 50000)])
def test_threads_of_candidates(rc, blocks, block, phases, kind):
    against_oracle(rc, crowd(blocks, block, phases, kind))


@pytest.mark.parametrize("kind", [W, A])
@pytest.mark.parametrize("blocks,block,hot", [(512, 256, 1), (4, 40000, 3)])
def test_hot_cells_among_candidates(rc, blocks, block, hot, kind):
    # the hot cells' buckets exceed the registers and hold thousands of candidates
    against_oracle(rc, crowd(blocks, block, 64, kind, hot))


@pytest.mark.parametrize("kind", [W, A])
@pytest.mark.parametrize("blocks,block,phases", [(9600, 256, 8), (80, 32768, 8), (45, 40000, 8)])
def test_one_pass_buckets(rc, blocks, block, phases, kind):
    # two tables of candidates in buckets of 7,000 to 10,000 keys
    against_oracle(rc, crowd(blocks, block, phases, kind))
