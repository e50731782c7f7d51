"""Append of prefill-sized calls that start anywhere inside a page: whole tiles are found wherever they begin."""
import numpy as np
import pytest
import torch

import paper_2608_23834_b200 as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,hkv", [(128, 1), (256, 3)])
@pytest.mark.parametrize("page", [16, 48])
@pytest.mark.parametrize("starts", [(0,), (15,), (1, 0, 8), (7, 31, 16, 5)])
def test_runs_at_any_offset_write_what_single_tokens_write(d, hkv, page, starts):
    """One call with a chunk per request, chunk r starting at position starts[r] of its first page, some tokens
    skipped, some scattered and one page beyond the arena; against calls of 64 tokens, which store token by token
    (compared with the oracle in test_gpu_lifecycle_kernels)."""
    rng = np.random.default_rng(sum(starts) + d + page)
    slots, first = [], 0
    for s in starts:
        n = int(rng.integers(280, 460))
        slots.append(first * page + s % page + np.arange(n))
        first += (s % page + n + page - 1) // page
    slots.append(first * page + rng.permutation(page))              # one page in random order
    first += 1
    slots = np.concatenate(slots).astype(np.int32)
    page_ids = rng.permutation(first)
    slots = (page_ids[slots // page] * page + slots % page).astype(np.int32)
    slots[rng.integers(0, len(slots), 5)] = -1                       # skipped tokens
    slots[40:40 + 20] = (first + 2) * page + np.arange(20) % page    # beyond the arena: flagged, not written
    n = len(slots)
    assert n >= 256
    k, v = (torch.from_numpy(rng.standard_normal((n, hkv, d)).astype(np.float32) * 50).cuda().to(torch.bfloat16) for _ in range(2))
    pools = [M.Pool(d, hkv, hkv, first, 1, np.ones(d, np.int8), page_tokens=page) for _ in range(2)]
    t = torch.from_numpy(slots).cuda()
    pools[0].append(k, v, t)
    for lo in range(0, n, 64):
        pools[1].append(k[lo:lo + 64].contiguous(), v[lo:lo + 64].contiguous(), t[lo:lo + 64].contiguous())
    torch.cuda.synchronize()
    assert pools[0].status() == M.E_BOUNDS and pools[1].status() == M.E_BOUNDS
    assert torch.equal(pools[0].fp8_arena, pools[1].fp8_arena) and bool(pools[0].fp8_arena.any())
