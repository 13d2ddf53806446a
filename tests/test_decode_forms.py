"""Which form of the decode kernel a batch of head dimension 64 takes, on both sides of the lines: seen in the size of its units, which
follows from the number of warps that share the pages."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps


def unit_pages(rows, ctx, kv_heads=8, group=1, sms=148):
    shape = ps.make_shape(kv_heads * group, kv_heads, 64)
    plan, _ = ps.ps_attn_plan(shape, np.full(rows, ctx - 1), np.ones(rows, dtype=np.int32), (ctx + 15) // 16, ps.ps_plan_opts(0, 0, sms))
    info = ps.ps_plan_get_info(plan)
    items = ps.ps_plan_get_items(plan)[0]
    ps.ps_plan_free(plan)
    assert sum(-(-int(e) // 16) - int(b) // 16 for b, e in items[:, 2:4]) == rows * kv_heads * ((ctx + 15) // 16)
    return info.decode_segment_tokens // 16


@pytest.mark.parametrize("rows,ctx,warps", [
    (512, 40, 24), (512, 240, 24), (512, 241, 12),  # 15 pages a row, 16
    (444, 240, 24), (443, 240, 12), (443, 144, 24), (443, 145, 12),  # two rows a warp, nine pages a row, ten
    (267, 80, 24), (266, 80, 12), (267, 81, 12),     # 1.2 rows a warp, five pages a row, six
    (333, 96, 24), (332, 96, 12),                   # 1.5 rows a warp
])
def test_many_short_rows_take_24_warps(rows, ctx, warps):
    pages = rows * 8 * ((ctx + 15) // 16)
    share = -(-pages // (148 * warps))
    assert unit_pages(rows, ctx) in ((max(4, share),) if warps == 24 else (max(4, share), max(4, share) + 1))


@pytest.mark.parametrize("rows,ctx", [(500, 130), (600, 128), (950, 114), (1100, 210)])
def test_24_warps_are_not_taken_beyond_the_built_in_scratch(rows, ctx):
    """Eight q heads a kv head: the partial rows of 24 warps would need more than ps_attn_run_static has, those of 12 do not."""
    shape = ps.make_shape(64, 8, 64)
    plan, need = ps.ps_attn_plan(shape, np.full(rows, ctx - 1), np.ones(rows, dtype=np.int32), (ctx + 15) // 16, ps.ps_plan_opts(0, 0, 148))
    items = ps.ps_plan_get_items(plan)[0]
    slots = items[items[:, 6] >= 0, 6]
    ps.ps_plan_free(plan)
    assert need <= ps.PS_STATIC_WORKSPACE_BYTES
    assert len(set(slots.tolist())) == len(slots)
    assert unit_pages(rows, ctx, group=8) > unit_pages(rows, ctx, group=1)


@pytest.mark.parametrize("rows,ctx,pages", [(30, 500, 5), (30, 1000, 9), (80, 480, 12)])
def test_small_units_are_not_rounded_to_whole_stages(rows, ctx, pages):
    assert unit_pages(rows, ctx) == pages


@pytest.mark.parametrize("heads,kv_heads,dim,dtype", [(32, 8, 128, 0), (64, 8, 128, 0), (8, 8, 64, 0), (4, 2, 64, 0), (32, 8, 128, 1)])
@pytest.mark.parametrize("sms,above", [(148, 128), (132, 128), (128, 128), (64, 64)])
def test_large_batches_of_decode_rows_alone_run_on_128_sms(heads, kv_heads, dim, dtype, sms, above):
    shape = ps.make_shape(heads, kv_heads, dim, 16, dtype)
    token = 2 * kv_heads * dim * 2
    ctx = int(0.75e9 / token / 300)

    def sized(prior, q_len):
        plan, _ = ps.ps_attn_plan(shape, prior, q_len, (max(prior) + max(q_len) + 15) // 16, ps.ps_plan_opts(0, 0, sms))
        info = ps.ps_plan_get_info(plan)
        ps.ps_plan_free(plan)
        return info.decode_sms

    assert sized([ctx - 1] * 300, [1] * 300) == sms
    assert sized([ctx] * 300, [1] * 300) == (above if dtype == 0 else sms)
    assert sized([20 * ctx] * 300, [1] * 300) == (above if dtype == 0 else sms)
