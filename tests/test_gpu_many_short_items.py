"""Batches of many short prefill items at head dimension 128, which go to the single-CTA kernel: on either side of the line
between the two kernels, with ragged lengths, rows of few keys and large scores, alone and beside decode rows."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from parity_util import compare, oracle_subset
from test_gpu_prefill_pair import run_and_compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,n,longest", [(gen.SHAPE_8B, 46, 64), (gen.SHAPE_8B, 48, 64), (gen.SHAPE_8B, 60, 300), (gen.SHAPE_LARGE, 30, 130),
                                             (gen.Shape(8, 8, 128), 50, 300), (gen.Shape(16, 8, 128), 70, 129)])
@pytest.mark.parametrize("exp", [0, 6])
def test_many_short_prompts(shape, n, longest, exp):
    rng = np.random.default_rng(1030 + n)
    q_len = rng.integers(9, longest + 1, n)
    b = gen.make_batch(shape, 1030, rng.integers(0, 200, n).tolist(), q_len.tolist())
    run_and_compare(b, np.where(np.arange(b.total_q) % 7 == 0, exp, 0), "%d prompts" % n)


@pytest.mark.parametrize("rows,ctx", [(6, 300), (150, 1500)])
def test_many_short_prompts_beside_decode_rows(rows, ctx):
    import torch
    from workloads.device import DeviceBatch

    rng = np.random.default_rng(1040)
    n = 60
    b = gen.make_batch(gen.SHAPE_8B, 1040, rng.integers(ctx // 2, ctx, rows).tolist() + rng.integers(0, 130, n).tolist(),
                       [1] * rows + rng.integers(20, 150, n).tolist())
    db = DeviceBatch(b)
    info = db.plan()
    assert info.n_prefill_items >= 2.5 * 148
    out, lse = db.run()
    db.pa.check()
    reqs = list(range(0, rows, max(1, rows // 12))) + list(range(rows, rows + n, 4))
    want, want_lse, packed, keys = oracle_subset(b, reqs, with_keys=True)
    compare(out, lse, want, want_lse, packed, what="beside %d rows" % rows, few_key_rows=True, keys=keys)
    for _ in range(3):
        again, lse2 = db.run()
        assert torch.equal(out.view(torch.int16), again.view(torch.int16)) and torch.equal(lse, lse2)
    db.pa.check()
