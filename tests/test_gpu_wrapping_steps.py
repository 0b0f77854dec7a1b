"""Reduced nests whose step times the point's number leaves the iterator's type
while the iterator stays inside: against the oracle, narrow and wide models."""
import pytest

import oracle
from workloads.spec import Access, Array, GLOBAL, Loop, Model, R, Stmt, W, bid, const, it, tid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("lo,step", [(-2_100_000_000, 1 << 21), (-2_147_000_000, (1 << 23) + 5), (-(3 << 60), 1 << 52),
                                     (-(1 << 61), (1 << 53) + 3), (-7, 2)])
def test_steps(monkeypatch, lo, step, wide):
    import paper_2503_08946_gb300 as rc
    monkeypatch.setenv("RC_JIT", "1")
    far = (1 << 50,) if wide else ()
    a = Array("a", GLOBAL, (97,) + far)
    at = lambda e: (e % 97,) + ((const(5),) if wide else ())
    st = [Stmt([Access(0, W, at(it(0) // step + 3 * tid.x))], loops=[Loop(lo, min(-lo, lo + 2000 * step), step), Loop(0, 2)],
               guards=[it(0) - lo - 5 * step, const(1) - bid.x]),
          Stmt([Access(0, R, at(it(0) + tid.x))], loops=[Loop(0, 5)])]
    m = Model((2, 1, 1), (33, 1, 1), [a], st, name=f"s{step}")
    h = rc.rc_model_create(m)
    assert rc.rc_model_layout(h)["wide"] == int(wide)
    got, exp = rc.check(h), oracle.check(m)
    assert (got.status, got.instances, got.racy_cells, got.witness) == (exp.status, exp.instances, exp.racy_cells, exp.witness)
