"""Plans that are freed without a scan, after others whose events were recorded
inside a graph: no error is left behind for the next call."""
import pytest

import synth
from oracle import reader as R
from oracle import writer as W

from gpu_util import assert_columns_equal, engine, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_unscanned_plan_after_a_graph(batch):
    from paper_2602_17335_gb300 import native as N
    from paper_2602_17335_gb300.scan import alloc_outputs, stream_handle
    eng = engine()
    data = W.write_file(synth.config2_table(6000, 2500, string_pool_size=200, zipf_k=300),
                        synth.config2_spec(2500, 4096, "UNCOMPRESSED", 1))
    dev, expect = to_dev(data), R.read_file(data)
    idx = eng.index([dev])
    plan, sizes = eng.plan(idx, None, 0, -1, N.PQ_SCAN_BATCHED if batch else N.PQ_SCAN_GRAPH)
    outs = alloc_outputs(sizes)
    if batch:
        b = N.pq_batch_create(eng.ctx, [plan], [[o.desc() for o in outs]], N.PQ_SCAN_GRAPH)
        N.pq_batch_launch(eng.ctx, b, stream_handle())
        N.check(N.pq_batch_wait(b), eng.ctx)
        N.pq_batch_free(b)
    else:
        eng.scan(plan, outs)
        assert eng.wait(plan, len(outs))[0] == N.PQ_OK
    assert_columns_equal(outs, expect)
    N.pq_free_plan(plan)
    for _ in range(3):  # with the first plan's events in other places
        unscanned, _ = eng.plan(idx, None, 0, -1, N.PQ_SCAN_BATCHED)
        N.pq_free_plan(unscanned)
        assert_columns_equal(eng.read([dev]), expect)
    N.pq_free_index(idx)
    eng.close()
