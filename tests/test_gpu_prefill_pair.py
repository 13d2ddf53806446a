"""The CTA-pair prefill kernel (head dimension 128) where its own branches can go wrong: items of one to seven key tiles
(its score buffers, the groups that begin an item and the stages wrap at three, three and four), ragged ends, several items
per pair, and rows whose softmax sums leave the range in which weights are taken without their row maximum, which are
computed again relative to it."""
import numpy as np
import pytest

import oracle
from workloads import gen

from parity_util import compare, kv_bits, q_bits

pytestmark = pytest.mark.gpu


def scaled(bits, exps):
    """bf16 bit patterns [T, H, d] times 2 ** exps[token]: exact, the exponent field moves."""
    f = (bits.astype(np.uint32) << 16).view(np.float32) * (2.0 ** np.asarray(exps, dtype=np.float32))[:, None, None]
    return (f.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)


def bf16_bits(x):
    u = np.ascontiguousarray(x, dtype=np.float32).view(np.uint32)
    return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)


def f32(bits):
    return (bits.astype(np.uint32) << 16).view(np.float32)


def on_device(bits):
    import torch

    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


def run_and_compare(batch, exps, what, plant=None, opts=None):
    """``plant``: changes request 0's K bit patterns [kv_len, Hkv, d], given them and q's; returns the positions changed."""
    import torch
    from workloads.device import DeviceBatch

    s = batch.shape
    db = DeviceBatch(batch)
    q = np.concatenate([q_bits(batch, r) for r in range(batch.n)])
    q = scaled(q, exps)
    db.q = on_device(q)
    ks, vs = zip(*[kv_bits(batch, r) for r in range(batch.n)])
    if plant:
        changed = plant(ks[0], q)
        db.q = on_device(q)
        for at in changed:
            db.pa.write(on_device(ks[0][at : at + 1]), on_device(vs[0][at : at + 1]), db.block_table[0], [at], [1], max_pages=batch.max_pages)
    info = db.plan(opts)
    assert info.n_prefill_items > 0
    out, lse = db.run()
    db.pa.check()
    kp = oracle.plain_pool(ks, batch.block_table, batch.num_pages, s.page_size)
    vp = oracle.plain_pool(vs, batch.block_table, batch.num_pages, s.page_size)
    rr = [r for r in range(batch.n) for _ in range(int(batch.q_len[r]))]
    rt = [i for r in range(batch.n) for i in range(int(batch.q_len[r]))]
    want, want_lse = oracle.attn_rows(q, kp, vp, batch.block_table, batch.prior, batch.q_len, s.n_q_heads, s.n_kv_heads, s.head_dim,
                                      s.page_size, rr, rt)
    keys = np.array([int(batch.prior[r]) + i + 1 for r, i in zip(rr, rt)])
    # Large scores make rows see a few keys in effect, however many they have: the outputs are single V values, bf16-rounded
    # (compare() scales its bound for such rows by the value).  lse: fp32 arithmetic on scores of up to 2^e times the plain
    # ones, whose products and sums over d = 128 are each good to a few units of 2^-24.
    peaked = (np.asarray(exps) > 1) | (plant is not None)
    compare(out, None, want, want_lse, what=what, few_key_rows=True, keys=np.where(peaked, 1, keys))
    err = np.abs(lse.cpu().numpy().astype(np.float64) - want_lse)
    assert (err <= 2e-3 + 1e-5 * np.abs(want_lse)).all(), "%s: lse off by %.3e" % (what, err.max())
    again, lse2 = db.run()
    assert torch.equal(out.view(torch.int16), again.view(torch.int16)) and torch.equal(lse, lse2)
    return np.linalg.norm(out.float().cpu().numpy().astype(np.float64) - want) / np.linalg.norm(want)


@pytest.mark.parametrize("prior,chunk", [(1500, 200), (0, 300), (300, 77)])
def test_peaked_rows_are_normalised_by_the_weights_that_pv_multiplies(prior, chunk):
    """With scores of standard deviation 8 a few keys have most of the weight.  Rounding the output to bf16 is a relative error
    of 1.66e-3 by itself, and a weight's rounding (2^-9 / sqrt(3) = 1.13e-3) counts for a fraction of that as long as it
    goes into the sum as well: sqrt(1.66^2 + (0.6 * 1.13)^2) = 1.8e-3.  Left out of the sum it counts in full, 2.0e-3 and
    more."""
    b = gen.make_batch(gen.SHAPE_8B, 940, [prior], [chunk])
    assert run_and_compare(b, np.full(b.total_q, 3), "peaked") <= 1.9e-3


@pytest.mark.parametrize("shape", [gen.SHAPE_8B, gen.SHAPE_LARGE, gen.Shape(16, 8, 128)])
@pytest.mark.parametrize("prior", [0, 1, 100, 127, 128, 250, 384, 511, 640, 777])
def test_items_of_one_to_seven_key_tiles(shape, prior):
    b = gen.make_batch(shape, 900 + prior, [prior, prior + 60], [40, 21])
    run_and_compare(b, np.zeros(b.total_q), "prior %d" % prior)


def test_many_short_items_per_pair():
    b = gen.make_batch(gen.SHAPE_8B, 950, [0] * 12, [500, 40, 33, 260, 130, 129, 128, 127, 65, 64, 63, 300])
    run_and_compare(b, np.zeros(b.total_q), "many short items")


@pytest.mark.parametrize("redo", [False, True])
def test_more_one_tile_items_per_pair_than_records_fit_its_ring(redo):
    """13 to 15 items of one key tile per pair; with ``redo`` every ninth token's rows are computed again as well.  (With a
    segment longer than any item: the planner would otherwise give so many short items to the single-CTA kernel.)"""
    import paper_2507_17769_b200 as ps

    b = gen.make_batch(gen.SHAPE_8B, 955, [0, 40] * 65, [64, 33] * 65)
    run_and_compare(b, np.where(np.arange(b.total_q) % 9 == 0, 9, 0) if redo else np.zeros(b.total_q), "one-tile items", opts=ps.ps_plan_opts(0, 4096, 0))


@pytest.mark.parametrize("every", [1, 3, 97])
@pytest.mark.parametrize("exp", [6, 9])
def test_rows_out_of_range_are_computed_again(every, exp):
    """Q times 2^6 gives scores of hundreds (weights overflow and underflow without the row maximum), 2^9 of thousands;
    ``every``: which tokens are scaled (all, a third, a few), so that items mix such rows with ordinary ones."""
    b = gen.make_batch(gen.SHAPE_8B, 960 + exp, [300, 0, 129], [130, 200, 70])
    exps = np.where(np.arange(b.total_q) % every == 0, exp, 0)
    run_and_compare(b, exps, "exp %d every %d" % (exp, every))


@pytest.mark.parametrize("segment", [0, 128, 256, 384, 512])
def test_pairs_whose_last_item_ends_on_a_full_key_tile(segment):
    """A pair's last record may be out before V of its last tiles has landed: their softmax does not wait for V unless the
    last tile is ragged.  Chunks whose keys end on a tile boundary, cold in L2, beside decode rows that keep the memory system
    busy; ``segment``: the planner's own cuts, or items of one to four full tiles."""
    import torch
    import paper_2507_17769_b200 as ps
    from workloads.device import DeviceBatch

    rng = np.random.default_rng(970)
    rows, chunks = 64, 16
    b = gen.make_batch(gen.SHAPE_8B, 970, rng.integers(3000, 5000, rows).tolist() + [64 + 256 * (8 + k) for k in range(chunks)],
                       [1] * rows + [64] * chunks)
    db = DeviceBatch(b)
    first = {}
    for k in list(range(chunks)) * 3:
        idx = list(range(rows)) + [rows + k]
        q = torch.cat([db.q[:rows], db.q[rows + 64 * k : rows + 64 * (k + 1)]])
        bt = db.block_table[idx].contiguous()
        info = db.pa.plan(b.prior[idx], b.q_len[idx], b.max_pages, ps.ps_plan_opts(0, segment, 0) if segment else None)
        assert info.n_prefill_items > 0
        ps.ps_plan_set_wait_limit(db.pa._plan, 200_000_000)
        out, lse = db.pa.run(q, bt)
        db.pa.check()  # (a wait that runs out is an error here)
        if k in first:
            assert torch.equal(out.view(torch.int16), first[k][0].view(torch.int16)) and torch.equal(lse, first[k][1])
        first[k] = (out, lse)
    db.pa.close()


@pytest.mark.parametrize("segment", [0, 4096])
@pytest.mark.parametrize("score", [50.0, 85.0, 104.0, 139.0, 173.0, 177.4, 355.0, 5000.0])
def test_one_key_with_a_large_score(score, segment):
    """Ordinary rows of some 2000 keys in which one key has nearly all the weight, orthogonal to the other rows of its item,
    so that nothing else takes the item's sums out of range.  A kv head each for positions all over a tile; 50 to 177.4 are 72
    to 256 in powers of two, where weights first overflow and exponent arithmetic without a bound would wrap."""
    import paper_2507_17769_b200 as ps

    b = gen.make_batch(gen.SHAPE_8B, 980, [2100], [16])
    places = [640 + c for c in (1, 2, 3, 5, 64 + 2, 64 + 3, 34, 35)]

    def plant(k, q):
        for g, at in enumerate(places):
            rows = f32(q[:, 4 * g : 4 * g + 4]).reshape(64, 128).astype(np.float64)
            want = np.zeros(64)
            want[(7 * g) % 64] = score * np.sqrt(128)
            k[at, g] = bf16_bits(np.linalg.lstsq(rows, want, rcond=None)[0])
        return places

    run_and_compare(b, np.zeros(b.total_q), "score %g" % score, plant, ps.ps_plan_opts(0, segment, 0) if segment else None)


@pytest.mark.parametrize("prior", [0, 90, 700])
@pytest.mark.parametrize("where,offset", [("all", 60.0), ("all", -60.0), ("all", 300.0), ("all", -300.0), ("sample", -40.0), ("sample", -66.0),
                                          ("sample", -72.0), ("sample", -300.0), ("sample", 300.0), ("first", 60.0), ("first", 100.0)])
def test_scores_away_from_the_rows_reference(where, offset, prior):
    """Scores moved by an offset on all keys, on the 32 of every tile of which the first tile's are a row's reference, or on
    the first key: weights are relative to the reference, and -72 below the others the sums leave their range."""
    b = gen.make_batch(gen.SHAPE_8B, 990, [prior], [150])
    unit = np.full(128, 128 ** -0.5)

    def along(x, to):  # x's component along `unit` set to `to`
        return bf16_bits(x + (to - x @ unit)[..., None] * unit)

    def plant(k, q):
        q[:] = along(f32(q).astype(np.float64), 16.0)
        kv = np.arange(k.shape[0])
        hit = np.ones_like(kv, dtype=bool) if where == "all" else (kv % 64 >= 32) & (kv % 128 < 64) if where == "sample" else kv == 0
        k[:] = along(f32(k).astype(np.float64), np.where(hit, offset * 128 ** 0.5 / 16, 0.0)[:, None])
        return kv

    run_and_compare(b, np.zeros(b.total_q), "%s %g" % (where, offset), plant)


@pytest.mark.parametrize("past", [0, 384])
def test_a_nan_key_reaches_the_rows_that_see_it(past):
    """A NaN in one key makes the output of every row that sees it NaN, wherever its column is; other rows
    are not touched.  ``past``: first position of the keys' tile (the second one some rows see and others do not)."""
    import torch
    from workloads.device import DeviceBatch

    b = gen.make_batch(gen.SHAPE_8B, 981, [300], [200])
    db = DeviceBatch(b)
    ks, vs = kv_bits(b, 0)
    places = [past + c for c in (1, 2, 3, 5, 66, 67, 34, 35)]
    db.plan()
    clean = db.run()[0]
    for g, at in enumerate(places):
        ks[at, g] = 0x7FC0
        db.pa.write(on_device(ks[at : at + 1]), on_device(vs[at : at + 1]), db.block_table[0], [at], [1], max_pages=b.max_pages)
    out, _ = db.run()
    db.pa.check()
    for g, at in enumerate(places):
        sees = torch.arange(300, 500, device="cuda") >= at
        heads = slice(4 * g, 4 * g + 4)
        assert bool(torch.isnan(out[sees][:, heads].float()).all()), "key %d" % at
        assert bool(torch.isfinite(out[~sees][:, heads].float()).all()), "key %d" % at
        if bool((~sees).any()):
            assert (out[~sees][:, heads].float() - clean[~sees][:, heads].float()).abs().max().item() <= 1e-2
