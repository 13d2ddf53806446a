"""The prefill kernel of head dimension 64 where its own branches can go wrong: q tiles of one to seven key tiles (its K and V
stages wrap at four, the phases of its one score tile and one weight tile a q tile at two), items of one q tile and of two that see different numbers of key
tiles, ragged ends, more items than its record ring holds, cut items of which a q tile sees nothing, and rows whose sums leave
the range in which weights are taken without their row maximum.  Oracle and bounds: those of the CTA-pair kernel's tests."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from test_gpu_prefill_pair import bf16_bits, f32, on_device, run_and_compare

pytestmark = pytest.mark.gpu

SHAPES = [gen.Shape(8, 8, 64), gen.Shape(4, 2, 64), gen.Shape(16, 2, 64)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prior", [0, 1, 100, 127, 128, 250, 384, 511, 640, 777])
def test_q_tiles_of_one_to_seven_key_tiles(shape, prior):
    chunks = [16 * 8 // (shape.n_q_heads // shape.n_kv_heads) * k // 4 for k in (3, 5, 8, 9)]  # 3/4, 5/4, 2 and 9/4 q tiles
    b = gen.make_batch(shape, 1900 + prior, [prior, prior + 60, prior, prior + 7], chunks)
    run_and_compare(b, np.zeros(b.total_q), "prior %d" % prior)


@pytest.mark.parametrize("segment", [128, 256, 384])
def test_cut_items(segment):
    b = gen.make_batch(gen.Shape(8, 8, 64), 1910, [0, 64, 300, 777], [256, 250, 257, 511])
    run_and_compare(b, np.zeros(b.total_q), "segment %d" % segment, opts=ps.ps_plan_opts(0, segment, 0))


@pytest.mark.parametrize("sms", [0, 3])
def test_more_items_than_records_fit_the_ring(sms):
    """With three SMs some 60 items a CTA: from a queue, of one q tile and of two."""
    b = gen.make_batch(gen.Shape(8, 8, 64), 1920, [0] * 18, [500, 40, 33, 260, 130, 129, 128, 127, 65, 64, 63, 300, 200, 9, 10, 255, 257, 256])
    run_and_compare(b, np.where(np.arange(b.total_q) % 9 == 0, 9, 0) if sms else np.zeros(b.total_q), "many items", opts=ps.ps_plan_opts(0, 0, sms))


@pytest.mark.parametrize("every", [1, 3, 97])
@pytest.mark.parametrize("exp", [6, 9])
def test_rows_out_of_range_are_computed_again(every, exp):
    b = gen.make_batch(gen.Shape(4, 2, 64), 1930 + exp, [300, 0, 129], [130, 200, 70])
    run_and_compare(b, np.where(np.arange(b.total_q) % every == 0, exp, 0), "exp %d every %d" % (exp, every))


@pytest.mark.parametrize("prior", [0, 90, 700])
@pytest.mark.parametrize("where,offset", [("all", 60.0), ("all", -300.0), ("sample", -66.0), ("sample", -72.0), ("sample", 300.0), ("first", 100.0)])
def test_scores_away_from_the_rows_reference(where, offset, prior):
    b = gen.make_batch(gen.Shape(8, 8, 64), 1990, [prior], [150])
    unit = np.full(64, 64 ** -0.5)

    def along(x, to):  # x's component along `unit` set to `to`
        return bf16_bits(x + (to - x @ unit)[..., None] * unit)

    def plant(k, q):
        q[:] = along(f32(q).astype(np.float64), 16.0)
        kv = np.arange(k.shape[0])
        hit = np.ones_like(kv, dtype=bool) if where == "all" else (kv % 64 >= 32) & (kv % 128 < 64) if where == "sample" else kv == 0
        k[:] = along(f32(k).astype(np.float64), np.where(hit, offset * 64 ** 0.5 / 16, 0.0)[:, None])
        return kv

    run_and_compare(b, np.zeros(b.total_q), "%s %g" % (where, offset), plant)


@pytest.mark.parametrize("prior,chunk", [(1500, 200), (0, 300), (300, 77)])
def test_peaked_rows_are_normalised_by_the_weights_that_pv_multiplies(prior, chunk):
    b = gen.make_batch(gen.Shape(8, 8, 64), 1940, [prior], [chunk])
    assert run_and_compare(b, np.full(b.total_q, 3), "peaked") <= 1.9e-3  # (derived at the pair kernel's test)


def test_a_nan_key_reaches_the_rows_that_see_it():
    import torch
    from workloads.device import DeviceBatch
    from parity_util import kv_bits

    b = gen.make_batch(gen.Shape(8, 8, 64), 1981, [300], [200])
    db = DeviceBatch(b)
    ks, vs = kv_bits(b, 0)
    places = [384 + c for c in (1, 2, 3, 5, 66, 67, 34, 35)]
    db.plan()
    for g, at in enumerate(places):
        ks[at, g] = 0x7FC0
        db.pa.write(on_device(ks[at : at + 1]), on_device(vs[at : at + 1]), db.block_table[0], [at], [1], max_pages=b.max_pages)
    out, _ = db.run()
    db.pa.check()
    for g, at in enumerate(places):
        sees = torch.arange(300, 500, device="cuda") >= at
        assert bool(torch.isnan(out[sees][:, g].float()).all()) and bool(torch.isfinite(out[~sees][:, g].float()).all()), "key %d" % at
