"""ps_attn_run inside a CUDA stream capture: the graph replays the plan bit for bit, and calls outside the capture
keep working afterwards."""
import pytest

import paper_2507_17769_b200 as ps
from workloads import gen

from parity_util import compare, oracle_subset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["decode rows", "mixed batch", "cut prefill items"])
def test_captured_run_replays_the_plan(which):
    import torch
    from workloads.device import DeviceBatch

    if which == "decode rows":
        b, opts = gen.make_batch(gen.SHAPE_8B, 3, [511, 2047, 15, 999], [1, 1, 1, 1]), None
    elif which == "mixed batch":
        b, opts = gen.config0(), None
    else:
        b, opts = gen.make_batch(gen.SHAPE_8B, 4, [700, 100], [40, 200]), ps.ps_plan_opts(0, 128, 0)
    db = DeviceBatch(b)
    db.plan(opts)
    eager, eager_lse = db.run()
    db.pa.check()
    want, want_lse, _ = oracle_subset(b, range(b.n))
    compare(eager, eager_lse, want, want_lse, what=which)

    out, lse = torch.zeros_like(eager), torch.zeros_like(eager_lse)
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        db.pa.run(db.q, db.block_table, out=out, lse=lse)
    for _ in range(3):
        out.zero_()
        lse.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, eager) and torch.equal(lse, eager_lse)
    db.pa.check()
    # calls outside the capture are not disturbed by it, whichever image slot they land on
    for _ in range(4):
        again, again_lse = db.run()
        db.pa.check()
        assert torch.equal(again, eager) and torch.equal(again_lse, eager_lse)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, eager)


@pytest.mark.parametrize("joined", [False, True])
def test_captured_append_and_gather_follow_the_kernels_that_make_their_inputs(joined):
    """Appends and gathers are launched early behind a kernel; in a graph they still wait for what they read, one producer or
    (``joined``) two on different branches, and what follows them waits for them."""
    import torch

    n, hkv, d = 700, 8, 128
    pa = ps.PagedAttention(32, hkv, d, 64, poison=True)
    bt = torch.randperm(64, device="cuda").to(torch.int32)[None].contiguous()
    src = torch.zeros((n, hkv, d), dtype=torch.bfloat16, device="cuda")
    k, v = torch.empty_like(src), torch.empty_like(src)
    other, side = torch.cuda.Stream(), torch.cuda.Stream()

    def step():
        if joined:
            other.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(other):
                for _ in range(20):
                    v.copy_(src).mul_(2)
        for _ in range(20):
            torch.add(src, 1, out=k)
        if joined:
            torch.cuda.current_stream().wait_stream(other)
        else:
            torch.mul(src, 2, out=v)
        pa.write(k, v, bt, [100], [n])
        gk, gv = pa.gather(bt[0], 100 + n)
        return gk[100:] + 0, gv[100:] + 0

    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        gk, gv = step()
    for i in range(1, 6):
        src.copy_(torch.randn_like(src))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(gk, src + 1) and torch.equal(gv, src * 2), "replay %d" % i
    pa.check_pool()
    pa.close()
