"""Decode batches too small for a share per warp, which run as a CTA per piece of a (row, kv head): rows around the sizes
at which a warp gets its next page (12 pages to a turn) and a row is cut (48 pages), the most rows and pages that still
run this way and the first that do not, group sizes 1 to 8.  Tolerance: that of the other parity tests."""
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from parity_util import compare, oracle_subset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [gen.Shape(8, 8, 64), gen.Shape(4, 2, 64), gen.Shape(8, 1, 128), gen.SHAPE_8B, gen.SHAPE_LARGE])
@pytest.mark.parametrize("ctx,sms,ctas", [
    ([1], 148, True), ([15, 16, 17, 191, 192, 193], 148, True), ([767, 768, 769, 385, 5], 148, True), ([12000, 1], 148, True),
    ([1536, 1535], 0, True),     # as many SMs as (row, kv head) pairs: uncut, eight pages a warp
    ([1537, 1], 0, False),       # and a piece of more than that: a share per warp
    ([40, 50, 60], -1, False),   # fewer SMs than pairs
])
def test_a_cta_per_piece(shape, ctx, sms, ctas):
    import torch
    from workloads.device import DeviceBatch

    b = gen.make_batch(shape, 9300 + len(ctx), [c - 1 for c in ctx], [1] * len(ctx))
    db = DeviceBatch(b, poison=True)
    pairs = len(ctx) * shape.n_kv_heads
    info = db.plan(ps.ps_plan_opts(0, 0, sms if sms > 0 else max(pairs + sms, 1)))
    assert (info.n_decode_items <= info.decode_sms and info.decode_segment_tokens >= 48 * 16) == ctas
    out, lse = db.run()
    db.pa.check()
    want, want_lse, _, keys = oracle_subset(b, range(b.n), with_keys=True)
    compare(out, lse, want, want_lse, what="ctx %s" % ctx, few_key_rows=True, keys=keys)
    out2, lse2 = db.run()
    db.pa.check()
    assert torch.equal(out.view(torch.int16), out2.view(torch.int16)) and torch.equal(lse, lse2)
