"""Append, gather and run of PagedAttention through the extension that takes tensors, against the same calls through addresses, which
tensors of subclasses still take: results, refusals, arguments given and left out."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

pytestmark = pytest.mark.gpu


def batch():
    from workloads.device import DeviceBatch

    b = gen.make_batch(gen.Shape(8, 2, 128), 9800, [99, 5, 40, 300], [1, 1, 20, 130])
    return b, DeviceBatch(b)


def test_results_and_arguments():
    import torch

    class Sub(torch.Tensor):
        pass

    b, db = batch()
    info = db.plan()
    assert isinstance(info, ps.binding.ps_plan_info)
    out, lse = db.run()
    assert out.shape == db.q.shape and out.dtype == db.q.dtype and lse.shape == (b.total_q, 8) and lse.dtype == torch.float32
    plain_out, plain_lse = db.pa.run(db.q.as_subclass(Sub), db.block_table)
    assert torch.equal(out.view(torch.int16), plain_out.view(torch.int16)) and torch.equal(lse, plain_lse)
    a, c = torch.empty_like(db.q), torch.empty_like(lse)
    got = db.pa.run(db.q, db.block_table, out=a, lse=c)
    assert got[0] is a and got[1] is c and torch.equal(a.view(torch.int16), out.view(torch.int16)) and torch.equal(c, lse)
    none = db.pa.run(db.q, db.block_table, want_lse=False)
    assert none[1] is None and torch.equal(none[0].view(torch.int16), out.view(torch.int16))
    assert db.pa.run(db.q, db.block_table, lse=c, want_lse=False)[1] is c
    db.pa.check()

    length = int(b.kv_len[3])
    k, v = db.pa.gather(db.block_table[3], length)
    k2, v2 = db.pa.gather(db.block_table[3].data_ptr(), np.int64(length))
    assert k.shape == (length, 2, 128) and k.is_contiguous() and k.dtype == torch.bfloat16
    assert torch.equal(k.view(torch.int16), k2.view(torch.int16)) and torch.equal(v.view(torch.int16), v2.view(torch.int16))
    empty = db.pa.gather(db.block_table[3], 0)
    assert empty[0].shape == (0, 2, 128)
    # appended again, with lengths of other types and max_pages given or not
    for prior, q_len, max_pages in (([0], [length], None), (np.array([0]), np.array([length]), b.max_pages), (np.array([[0, 7]], dtype=np.int32)[:, 0], (length,), None)):
        for cast in (lambda x: x, lambda x: x.as_subclass(Sub)):
            db.pa.write(cast(v), cast(k), db.block_table[3:4], prior, q_len, max_pages)
            k2, v2 = db.pa.gather(db.block_table[3], length)
            assert torch.equal(k.view(torch.int16), v2.view(torch.int16)) and torch.equal(v.view(torch.int16), k2.view(torch.int16))
            k, v = k2, v2
    db.pa.check_pool()


def test_refusals():
    import torch

    b, db = batch()
    db.plan()
    wide = torch.empty((b.total_q, 16, 128), dtype=torch.bfloat16, device="cuda")
    for q, bt in ((db.q[:-1], db.block_table), (wide[:, ::2], db.block_table), (db.q, db.block_table.t().contiguous().t())):
        with pytest.raises(AssertionError):
            db.pa.run(q, bt)
    with pytest.raises(AssertionError):
        db.pa.write(wide[:1, ::8], wide[:1, :2].contiguous(), db.block_table[:1], [0], [1])
    k = torch.zeros((1, 2, 128), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ps.PsError) as e:
        db.pa.write(k, k, db.block_table[:1], [-1], [1])
    assert e.value.status == ps.binding.PS_ERR_INVALID
    with pytest.raises(ValueError):
        db.pa.write(k, k, db.block_table[:1], [0, 0], [1])
    with pytest.raises(RuntimeError):
        db.pa.gather(db.block_table[0], -1)
    with pytest.raises(OverflowError):
        db.pa.write(k, k, db.block_table[:1], [0], [1], max_pages=1 << 40)
    fp8 = ps.PagedAttention(8, 2, 128, 4, kv_dtype=1)
    with pytest.raises(AssertionError):
        fp8.gather(db.block_table[0], 1)
    other = ps.PagedAttention(8, 2, 64, b.num_pages)
    other.plan(b.prior, b.q_len, b.max_pages)
    db.pa._plan, plan = other._plan, db.pa._plan
    with pytest.raises(ps.PsError):  # (plan and pool of different shapes)
        db.pa.run(db.q, db.block_table)
    db.pa._plan = plan
    out, _ = db.run()
    db.pa.check()
    assert bool(torch.isfinite(out.float()).all())
