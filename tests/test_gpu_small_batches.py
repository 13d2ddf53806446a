"""Small batches, whose work lists travel as kernel parameters: the status words of their runs, which the library keeps for a
limited number of plans and hands from a freed plan to the next.  And batches whose two kernels are launched on one stream: what
per-kernel timing reports of them."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps
from paper_2507_17769_b200 import binding as B
from workloads import gen

pytestmark = pytest.mark.gpu


def small():
    from workloads.device import DeviceBatch

    return DeviceBatch(gen.make_batch(gen.SHAPE_8B, 1010, [400, 33, 900], [1, 1, 40]))


def test_a_status_word_given_back_reports_for_its_next_plan_only():
    import torch

    db = small()
    want = db.plan() and db.run()
    db.pa.check()
    stream = torch.cuda.current_stream().cuda_stream
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    bad = db.block_table.clone()
    bad[0, 0] = db.batch.num_pages  # outside the pool: skipped by the kernel, and reported

    def run(table):
        plan, _ = ps.ps_attn_plan(db.pa.shape, db.batch.prior, db.batch.q_len, db.batch.max_pages)
        out, lse = torch.empty_like(want[0]), torch.empty_like(want[1])
        B.ps_attn_run(plan, db.pa.kv, db.q, table, out, lse, ws, ws.numel(), stream)
        try:
            B.ps_plan_status(plan, stream)
            return out, lse
        finally:
            ps.ps_plan_free(plan)

    for k in range(4):
        with pytest.raises(ps.PsError) as e:
            run(bad)
        assert e.value.status == B.PS_ERR_BOUNDS
        out, lse = run(db.block_table)
        assert torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse, want[1])


def test_more_plans_alive_than_status_words():
    import torch

    db = small()
    want = db.plan() and db.run()
    stream = torch.cuda.current_stream().cuda_stream
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    bad = db.block_table.clone()
    bad[0, 0] = -1
    plans = []
    try:
        for _ in range(300):
            plans.append(ps.ps_attn_plan(db.pa.shape, db.batch.prior, db.batch.q_len, db.batch.max_pages)[0])
        for plan in (plans[0], plans[200], plans[270], plans[299]):
            out, lse = torch.empty_like(want[0]), torch.empty_like(want[1])
            B.ps_attn_run(plan, db.pa.kv, db.q, bad, out, lse, ws, ws.numel(), stream)
            with pytest.raises(ps.PsError) as e:
                B.ps_plan_status(plan, stream)
            assert e.value.status == B.PS_ERR_BOUNDS
            B.ps_attn_run(plan, db.pa.kv, db.q, db.block_table, out, lse, ws, ws.numel(), stream)
            B.ps_plan_status(plan, stream)
            assert torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse, want[1])
    finally:
        for plan in plans:
            ps.ps_plan_free(plan)


@pytest.mark.parametrize("rows,ctx,chunk", [(32, 2000, 256), (16, 4000, 96)])
def test_recording_times_leaves_the_kernels_side_by_side(rows, ctx, chunk):
    """The two kernels' recorded intervals overlap as the kernels of a run that is not recorded do: recorded one after the
    other, a run takes more than their sum.  Outputs are the same."""
    import torch
    from workloads.device import DeviceBatch

    rng = np.random.default_rng(1020)
    db = DeviceBatch(gen.make_batch(gen.SHAPE_8B, 1020, rng.integers(ctx * 3 // 4, ctx * 5 // 4, rows).tolist() + [2000], [1] * rows + [chunk]))
    info = db.plan()
    assert info.decode_sms + info.prefill_sms == torch.cuda.get_device_properties(0).multi_processor_count and info.n_launches == 2
    want = db.run()
    runs, total = 20, []
    ps.ps_plan_set_timing(db.pa._plan, runs)
    for _ in range(runs):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        out, lse = db.run()
        e1.record()
        torch.cuda.synchronize()
        total.append(e0.elapsed_time(e1))
    prefill, decode, _, n = ps.ps_plan_get_timing(db.pa._plan, torch.cuda.current_stream().cuda_stream)
    db.pa.check()
    assert n == runs and torch.equal(out.view(torch.int16), want[0].view(torch.int16)) and torch.equal(lse, want[1])
    assert np.median(total) < prefill + decode, (np.median(total), prefill, decode)
