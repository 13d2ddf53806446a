"""ps_kv_write at the batch sizes where the lengths change the way they travel (kernel parameters of 64, 512 and 4000
requests, device memory beyond): every new token lands in its page, bit for bit, and nothing else is touched."""
import numpy as np
import pytest

import paper_2507_17769_b200 as ps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("n", [1, 64, 65, 512, 513, 4000, 4001])
def test_every_token_lands_in_its_page(n, fp8):
    import torch

    heads, dim, max_pages = 2, 128, 2
    rng = np.random.default_rng(n)
    q_len = rng.integers(1, 4, n).astype(np.int32)
    prior = rng.integers(0, 29, n).astype(np.int32)
    table = rng.permutation(2 * n).astype(np.int32).reshape(n, max_pages)
    pa = ps.PagedAttention(heads, heads, dim, 2 * n, kv_dtype=int(fp8))
    pa.pool.zero_()
    bt = torch.from_numpy(table).cuda()
    g = torch.Generator(device="cuda").manual_seed(n)
    k, v = (torch.randn((int(q_len.sum()), heads, dim), generator=g, device="cuda").bfloat16() for _ in range(2))
    pa.write(k, v, bt, prior, q_len)
    pa.check_pool()
    start = np.concatenate([[0], np.cumsum(q_len)])
    for r in sorted({0, n // 3, n // 2, n - 1} | set(rng.integers(0, n, 8).tolist())):
        new = slice(int(start[r]), int(start[r + 1]))
        pos = slice(int(prior[r]), int(prior[r] + q_len[r]))
        if fp8:
            kc, vc, ks, vs = pa.gather_fp8(bt[r], 32)
            for codes, scale, x in ((kc, ks, k), (vc, vs, v)):
                # a code is within half a step (2^-4 of the value, or of the smallest normal 2^-6) of what it stands for
                x, scale = x[new].float(), scale[pos][..., None]
                got = codes[pos].view(torch.float8_e4m3fn).float() * scale
                assert bool(((got - x).abs() <= torch.maximum(x.abs(), scale * 2.0 ** -6) * 2.0 ** -4).all())
                rest = torch.ones(32, dtype=torch.bool)
                rest[pos] = False
                assert int(codes[rest.cuda()].sum()) == 0
        else:
            for got, x in zip(pa.gather(bt[r], 32), (k, v)):
                assert torch.equal(got[pos].view(torch.int16), x[new].view(torch.int16))
                rest = torch.ones(32, dtype=torch.bool)
                rest[pos] = False
                assert float(got[rest.cuda()].float().abs().sum()) == 0.0


@pytest.mark.parametrize("heads,dim", [(1, 64), (3, 64), (8, 64), (20, 64), (1, 128), (8, 128), (9, 128), (20, 128)])
@pytest.mark.parametrize("aligned", [True, False])
def test_append_and_gather_move_every_byte_of_a_row(heads, dim, aligned):
    """Rows of fewer, as many and more 32-byte pairs than a warp moves at a time, in tensors that start at a 32-byte
    boundary or only at a 16-byte one: what was appended (behind an odd and an even slot) is read back bit for bit."""
    import torch

    pa = ps.PagedAttention(heads, heads, dim, 32, poison=True)
    bt = torch.randperm(32, device="cuda", dtype=torch.int32).reshape(2, 16)
    q_len, prior = np.array([37, 9], dtype=np.int32), np.array([0, 0], dtype=np.int32)
    g = torch.Generator(device="cuda").manual_seed(heads * dim)

    def place(n):
        room = torch.empty(n * heads * dim + 16, device="cuda", dtype=torch.bfloat16)
        return room[0 if aligned else 8:][: n * heads * dim].view(n, heads, dim)

    def tokens(n):
        x = place(n)
        x.copy_(torch.randn((n, heads, dim), generator=g, device="cuda"))
        return x

    parts = [(tokens(46), tokens(46)), (tokens(4), tokens(4))]
    pa.write(*parts[0], bt, prior, q_len)
    pa.write(*parts[1], bt, q_len, np.array([1, 3], dtype=np.int32))
    pa.check_pool()
    for r, (old, new) in enumerate(((slice(0, 37), slice(0, 1)), (slice(37, 46), slice(1, 4)))):
        n = int(q_len[r]) + (1, 3)[r]
        outs = (place(n), place(n))
        ps.ps_kv_gather(pa.kv, bt[r].data_ptr(), n, outs[0].data_ptr(), outs[1].data_ptr(), torch.cuda.current_stream().cuda_stream)
        for got, a, b in zip(outs, parts[0], parts[1]):
            assert torch.equal(got.view(torch.int16), torch.cat([a[old], b[new]]).view(torch.int16))
