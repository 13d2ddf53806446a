"""Decode at head dimension 64 with a unit per warp, two pages to a stage: rows and units that end in an odd page (the stage's second
half then holds an older page), in the middle of a page and on its edge, with groups of 1 to 8 heads.  Tolerance: that of the
other parity tests."""
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from parity_util import compare, oracle_subset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [gen.Shape(8, 8, 64), gen.Shape(4, 2, 64), gen.Shape(8, 2, 64), gen.Shape(16, 2, 64)])
@pytest.mark.parametrize("segment", [16, 32, 48, 80, 0])
def test_two_pages_a_stage(shape, segment):
    import torch
    from workloads.device import DeviceBatch

    ctx = [1, 15, 16, 17, 32, 33, 47, 48, 49, 64, 65, 513, 527, 529, 1000, 1025]
    b = gen.make_batch(shape, 9700, [c - 1 for c in ctx], [1] * len(ctx))
    db = DeviceBatch(b, poison=True)
    info = db.plan(ps.ps_plan_opts(segment, 0, 0 if segment else 2))
    assert segment == 0 or info.decode_segment_tokens == segment
    out, lse = db.run()
    db.pa.check()
    want, want_lse, _, keys = oracle_subset(b, range(b.n), with_keys=True)
    compare(out, lse, want, want_lse, what="segment %d" % segment, few_key_rows=True, keys=keys)
    out2, lse2 = db.run()
    db.pa.check()
    assert torch.equal(out.view(torch.int16), out2.view(torch.int16)) and torch.equal(lse, lse2)


@pytest.mark.parametrize("shape", [gen.Shape(8, 8, 64), gen.Shape(32, 8, 64)])
@pytest.mark.parametrize("last", [1, 15, 16, 17, 33])
def test_a_page_a_stage_for_many_short_rows(shape, last):
    """Units that span several rows, rows that end in the middle of a page and on its edge, rows cut between two warps."""
    import torch
    from workloads.device import DeviceBatch

    ctx = [32 + (7 * k + last) % 17 for k in range(310)] + [last, 200, 1, 160]
    b = gen.make_batch(shape, 9710 + last, [c - 1 for c in ctx], [1] * len(ctx))
    db = DeviceBatch(b, poison=True)
    assert db.plan().decode_segment_tokens == 64  # (the share of 24 warps an SM)
    out, lse = db.run()
    db.pa.check()
    want, want_lse, _, keys = oracle_subset(b, range(b.n), with_keys=True)
    compare(out, lse, want, want_lse, what="last %d" % last, few_key_rows=True, keys=keys)
    out2, lse2 = db.run()
    db.pa.check()
    assert torch.equal(out.view(torch.int16), out2.view(torch.int16)) and torch.equal(lse, lse2)
