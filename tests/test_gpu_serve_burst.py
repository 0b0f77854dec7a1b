"""A burst of requests is batched: the server does not keep the submitting thread
out while it enqueues a batch or reads one back."""
import statistics

import pytest

import workloads as w

pytestmark = pytest.mark.gpu


def test_burst_is_batched():
    import paper_2503_08946_gb300 as rc
    handles = [rc.rc_model_create(m) for m in w.batch_models(500, seed0=11, t_max=2048)]
    mean = []
    for _ in range(5):
        srv = rc.RcServer(memory_bytes=2 << 30, slots=4)
        try:
            ids = [srv.submit(handles[i % 500]) for i in range(2000)]
            done = []
            while len(done) < len(ids):
                done += srv.poll(1024, 100)
        finally:
            srv.close()
        assert sorted(d.request for d in done) == sorted(ids)
        mean.append(len(done) / sum(1.0 / d.batch_size for d in done))
    # batches of 3 when every submission waited for the enqueueing of a batch
    assert statistics.median(mean) >= 6, mean
