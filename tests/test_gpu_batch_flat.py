"""The flat batch expansion (loop-free models with one-dimensional grids and blocks):
one and four model threads per lane, at thread counts around its units, with guards, terms of every kind, table loads, out-of-bounds reports and
scopes; each result against the oracle."""
import pytest

import oracle
from workloads.rng import SplitMix64
from workloads.spec import A, Access, Array, GLOBAL, Loop, Model, R, SHARED, Stmt, W, bid, const, load, tid

pytestmark = pytest.mark.gpu
T = [1, 31, 33, 127, 128, 129, 511, 512, 513, 640, 1025, 2000]


@pytest.fixture(scope="module")
def rc():
    import torch
    import paper_2503_08946_gb300 as m
    assert torch.cuda.is_available()
    return m


def model(seed, threads, big=0, oob=False, tables=True):
    rng = SplitMix64(0xF1A7 ^ seed * 0x9E3779B97F4A7C15)
    block = (32, 48, 96, 100, 256)[rng.below(5)]
    nb = (threads + block - 1) // block
    g = bid.x * block + tid.x
    s, a = Array("s", SHARED, (64, 3)), Array("g", GLOBAL, (777,))
    st = []
    for k in range(rng.uniform_int(1, 6)):
        e = rng.uniform_int(-5, 5) * tid.x + rng.uniform_int(-3, 3) * bid.x + const(rng.uniform_int(-40, 40) + big)
        d = (1, 2, 3, 7, 32, 1000, 65537)[rng.below(7)]
        e = e // d if rng.chance(0.5) else e % d + rng.uniform_int(-2, 2) * tid.x
        if tables and rng.chance(0.2):
            e = e + load(0, tid.x % 5)
        acc = [Access(1, (R, W, A)[rng.below(3)], (e % 777,))]
        if rng.chance(0.5):
            acc.append(Access(0, (R, W)[rng.below(2)], (e % 64, tid.x % 3)))
        if oob and k == 0:
            acc.append(Access(1, W, (g + (777 - threads + 1),)))
        st.append(Stmt(acc, guards=[const(threads - 1) - g] + ([e % 5 - 1] if rng.chance(0.4) else []),
                       phase=(bid.x + k) % 3, warp_phase=const(0)))
    return Model((nb, 1, 1), (block, 1, 1), [s, a], st, n_phases=3, tables=[[4, -7, 0, 9, 2]] if tables else [],
                 name=f"flat{seed}_{threads}")


def run(rc, models):
    h = [rc.rc_model_create(m) for m in models]
    got = rc.rc_report(rc.rc_check_batch(h, None, rc.workspace(rc.rc_batch_workspace_size(h, None))))
    for m, r in zip(models, got):
        e = oracle.check(m)
        assert (r.status, r.instances) == (e.status, e.instances), (m.name, r, e)
        if e.status:
            assert (r.oob_stmt, r.oob_access, r.oob_gtid, r.oob_dim) == (e.oob_stmt, e.oob_access, e.oob_gtid, e.oob_dim)
        else:
            assert (r.verdict, r.racy_cells, r.witness) == (e.verdict, e.racy_cells, e.witness), m.name


@pytest.mark.parametrize("tables", [False, True])
@pytest.mark.parametrize("seed", range(4))
def test_one_thread_per_lane(rc, seed, tables):
    run(rc, [model(100 * seed + i, t, tables=tables) for i, t in enumerate(T)])


@pytest.mark.parametrize("tables", [False, True])
@pytest.mark.parametrize("seed", range(2))
def test_four_threads_per_lane(rc, seed, tables):
    # enough units of 512 threads for the wide kernel: 30 models of 20,000 to 34,000 threads
    run(rc, [model(10000 * seed + i, 20000 + 467 * i, tables=tables) for i in range(30)] +
            [model(10100 * seed + i, t, tables=tables) for i, t in enumerate(T)])


@pytest.mark.parametrize("big", [(1 << 31) - 3000, -(1 << 31) + 3000, (1 << 31) + 5, 1 << 40])
def test_values_around_32_bits(rc, big):
    run(rc, [model(7000 + i, t, big=big, tables=False) for i, t in enumerate(T)])


def test_out_of_bounds_models_among_others(rc):
    run(rc, [model(9000 + i, t, oob=i % 3 == 0 and t <= 777, tables=False) for i, t in enumerate(T * 3)])
