"""Pages that go through append, demote, promote, demote and decode again and again without a synchronisation: every
call must see what the calls before it in the stream have written, although kernels start before their predecessors end."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_23834_b200 as M

pytestmark = pytest.mark.gpu

ROUNDS = 24


def _rounds(d, hkv, page, n, fmt, sync):
    """ROUNDS outputs of a decode over pages that were rewritten in every round, and the pool of the last round."""
    group, dev = 4, "cuda:0"
    sigma = (np.random.default_rng(d).integers(0, 2, d) * 2 - 1).astype(np.int8)
    pool = M.Pool(d, hkv, hkv * group, 2 * n, 2 * n, sigma, max_batch=n, page_tokens=page, tq3_format=fmt)
    gen = torch.Generator(device=dev).manual_seed(3)
    kv = [torch.randn((2, n * page, hkv, d), generator=gen, device=dev, dtype=torch.bfloat16) for _ in range(ROUNDS)]
    q = torch.randn((n, hkv * group, d), generator=gen, device=dev, dtype=torch.bfloat16)
    slots = torch.arange(n * page, dtype=torch.int32, device=dev)
    first, second = torch.arange(n, dtype=torch.int32, device=dev), torch.arange(n, 2 * n, dtype=torch.int32, device=dev)
    # row b: page b of the first TQ3 pages, of the promoted FP8 pages, and of the second TQ3 pages; ids and tags published
    bt = torch.full((n, 3), -1, dtype=torch.int32, device=dev)
    tags = torch.zeros((n, 3), dtype=torch.uint8, device=dev)
    entries = [torch.arange(n, device=dev) * 3 + i for i in range(3)]
    lens = torch.full((n,), 3 * page, dtype=torch.int32, device=dev)
    outs = [torch.empty((n, hkv * group, d), device=dev) for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for r in range(ROUNDS):
        steps = [lambda: pool.append(kv[r][0], kv[r][1], slots),
                 lambda: pool.demote(first, first, bt, tags, entries[0]),
                 lambda: pool.promote(first, second, bt, tags, entries[1]),
                 lambda: pool.demote(second, second, bt, tags, entries[2]),
                 lambda: pool.decode_attention(q, bt, tags, lens, d ** -0.5, out=outs[r])]
        for step in steps:
            step()
            if sync:
                torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert pool.status() == M.OK
    return outs, pool, sigma


@pytest.mark.parametrize("d,hkv,page,n,fmt", [(128, 8, 16, 5, 2), (128, 2, 16, 160, 1), (256, 4, 16, 5, 1), (256, 4, 16, 200, 2),
                                              (256, 2, 64, 3, 2), (128, 4, 1792, 2, 1)])
def test_recycled_pages_without_synchronisation(d, hkv, page, n, fmt):
    got, pool, sigma = _rounds(d, hkv, page, n, fmt, sync=False)
    want, _, _ = _rounds(d, hkv, page, n, fmt, sync=True)
    for r in range(ROUNDS):
        assert torch.equal(got[r], want[r]), r
    if page > 16:
        return
    with oracle.record_format(fmt):
        for p in (0, n - 1):
            fp8, tq3 = pool.page_read_raw(M.FMT_FP8, p).reshape(hkv, -1), pool.page_read_raw(M.FMT_TQ3, p).reshape(hkv, -1)
            back, again = pool.page_read_raw(M.FMT_FP8, n + p).reshape(hkv, -1), pool.page_read_raw(M.FMT_TQ3, n + p).reshape(hkv, -1)
            for h in range(hkv):
                assert np.array_equal(tq3[h], oracle.demote_record(fp8[h], d, sigma))
                assert np.array_equal(back[h], oracle.promote_record(tq3[h], d, sigma))
                assert np.array_equal(again[h], oracle.demote_record(back[h], d, sigma))
