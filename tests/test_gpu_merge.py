"""The merge kernel's two forms (four rows a warp where no item has more than four segments, else one): numbers of segments around the
line and around those that a warp's lanes hold, rows that are no multiple of four.  Tolerance: that of the other parity tests."""
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from parity_util import compare, oracle_subset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [gen.Shape(8, 8, 64), gen.Shape(4, 2, 64), gen.Shape(2, 2, 128), gen.SHAPE_8B])
@pytest.mark.parametrize("segments", [2, 3, 4, 5, 8, 9, 32, 33])
def test_segments(shape, segments):
    import torch
    from workloads.device import DeviceBatch

    b = gen.make_batch(shape, 9900 + segments, [128 * segments - 7, 128 * segments - 61], [7, 33])
    db = DeviceBatch(b, poison=True)
    info = db.plan(ps.ps_plan_opts(0, 128, 0))
    assert info.n_merge_rows == b.total_q * shape.n_q_heads
    out, lse = db.run()
    db.pa.check()
    want, want_lse, _ = oracle_subset(b, range(b.n))
    compare(out, lse, want, want_lse, what="%d segments" % segments)
    out2, lse2 = db.run()
    db.pa.check()
    assert torch.equal(out.view(torch.int16), out2.view(torch.int16)) and torch.equal(lse, lse2)


@pytest.mark.parametrize("shape,prior,q_len", [
    (gen.Shape(8, 8, 64), [900] * 20 + [2100, 700], [1] * 20 + [300, 500]),
    (gen.Shape(8, 8, 64), [900] * 24 + [2500], [1] * 24 + [200]),
    (gen.Shape(8, 2, 128), [1999] * 30 + [6000], [1] * 30 + [300]),
    (gen.Shape(8, 2, 128), [2499] * 60 + [3000], [1] * 60 + [200]),  # (the decode kernel ends last: merged under it)
    (gen.Shape(4, 2, 64), [1499] * 150 + [5000], [1] * 150 + [300]),
], ids=["d64-118-items", "d64-48-items", "d128", "d128-decode-last", "d64-decode-last"])
def test_mixed_batches_with_cut_items_back_to_back(shape, prior, q_len):
    """Decode, prefill and merge kernel on one stream, each launched while the one before it runs, or on two, for queries that change from
    run to run: bit for bit what a run gives whose kernels are recorded (decode kernel on a second stream) and one replayed from a graph."""
    import torch
    from workloads.device import DeviceBatch

    b = gen.make_batch(shape, 9950, prior, q_len)
    db = DeviceBatch(b, poison=True)
    info = db.plan()
    assert info.n_launches == 3 and info.decode_sms + info.prefill_sms <= 148  # (side by side, with a merge kernel)
    queries = [db.q, db.q.flip(0).contiguous()]
    got = []
    for k in range(20):  # no synchronisation inside this loop
        got.append(db.pa.run(queries[k % 2], db.block_table))
    db.pa.check()
    want, want_lse, _ = oracle_subset(b, range(b.n))
    compare(*got[0], want, want_lse, what="first run")
    graph_out = torch.empty_like(db.q), torch.empty_like(got[0][1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        db.pa.run(db.q, db.block_table, out=graph_out[0], lse=graph_out[1])
    graph.replay()
    db.pa.check()
    del graph
    ps.ps_plan_set_timing(db.pa._plan, 2)
    recorded = [db.pa.run(q, db.block_table) for q in queries]
    db.pa.check()
    ps.ps_plan_set_timing(db.pa._plan, 0)
    for k, (out, lse) in enumerate(got + [graph_out]):
        ref_out, ref_lse = recorded[k % 2]
        assert torch.equal(out.view(torch.int16), ref_out.view(torch.int16)) and torch.equal(lse, ref_lse), "run %d" % k
