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
