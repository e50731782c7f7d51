"""Batches in which a request of one to three pages stands beside long ones: every row is written by every call that cuts a
layer by itself, and the workspace is left as the next call needs it."""
import numpy as np
import pytest
import torch

import mkv_workloads as W
import oracle
import paper_2608_23834_b200 as M
from _gpu_util import Case, check_close

pytestmark = pytest.mark.gpu

LENS = (4000, 32, 2098, 25, 36, 2846, 3000, 40, 3000, 16000, 17)
BATCHES = [(0, 1), (2, 3), (4, 5), (6, 7, 8), (1, 9), (9, 1, 10), (3, 10, 0, 4)]


def _tickets(pool):
    """One arrival counter per possible block, behind the 256 reserved bytes of the workspace."""
    return pool.workspace[256:256 + 4 * 512].view(torch.int32)


def _calls(pools, c, at, out, lse):
    """The calls of one batch, each with the number of outputs that it writes."""
    q, bt, tags, lens, scale = c.q[at].contiguous(), c.bt[at].contiguous(), c.tags[at].contiguous(), c.lens[at].contiguous(), c.spec.scale
    layers = lambda n: M.decode_attention_layers(pools[:n], [q] * n, [bt] * n, [tags] * n, lens, scale, out[:n], lse[:n])
    yield "single", 1, lambda: pools[0].decode_attention(q, bt, tags, lens, scale, out=out[0], lse=lse[0])
    yield "static", 1, lambda: M.decode_attention_static(pools[0], q, bt, tags, lens, scale, out=out[0], lse=lse[0])
    yield "scored", 1, lambda: pools[0].decode_attention_scored(q, bt, tags, lens, scale, out=out[0], lse=lse[0])
    yield "two layers", 2, lambda: layers(2)
    yield "three layers", 3, lambda: layers(3)


@pytest.mark.parametrize("fmt", [1, 2])
@pytest.mark.parametrize("d,hkv,group", [(256, 1, 6), (256, 2, 4), (256, 4, 6), (128, 1, 8), (128, 2, 4)])
def test_a_short_row_beside_long_ones(d, hkv, group, fmt):
    with oracle.record_format(fmt):
        case = Case(W.config(0, seq_lens=LENS, head_dim=d, n_kv_heads=hkv, group=group, anchor_prefix=16, recent_tokens=300))
        ref, ref_lse = case.reference()
    pools = [case.pool]
    for _ in range(2):
        pools.append(M.Pool(d, hkv, hkv * group, max(case.tab.fp8_pages, 1), max(case.tab.tq3_pages, 1), case.L.sigma,
                            max_batch=len(LENS), tq3_format=fmt))
        pools[-1].upload_arenas(case.L.fp8_arena, case.L.tq3_arena)
    first = {}
    for turn in range(2):                     # every batch twice on the same workspaces, the others between
        for batch in BATCHES:
            at = torch.tensor(batch, device="cuda:0")
            new = lambda *shape: torch.full(shape, float("nan"), device="cuda:0")
            out, lse = [new(len(batch), hkv * group, d) for _ in range(3)], [new(len(batch), hkv * group) for _ in range(3)]
            for name, n, call in _calls(pools, case, at, out, lse):
                for o, l in zip(out, lse):
                    o.fill_(float("nan"))
                    l.fill_(float("nan"))
                call()
                torch.cuda.synchronize()
                for i in range(n):
                    what = f"{name}, layer {i}, batch {batch}, turn {turn}"
                    got, got_lse = out[i].cpu().numpy(), lse[i].cpu().numpy()
                    for k, b in enumerate(batch):
                        check_close(got[k], ref[b], what)
                        assert np.abs(got_lse[k] - ref_lse[b]).max() < 2e-3, what
                    assert np.array_equal(got, first.setdefault((name, i, batch), got)), what
                    assert not _tickets(pools[i]).any(), what
    assert all(p.status() == M.OK for p in pools)


def test_tables_of_more_positions_than_one_launch_counts():
    """300 requests x 128 heads in tables of 65,535 pages a row may hold 2^31 pages and more: the call takes several launches
    and gives what it gives for the same requests in a narrow table."""
    d, hkv, B, wide = 128, 128, 300, 65535
    rng = np.random.default_rng(5)
    lens = torch.from_numpy(rng.integers(0, 65, B).astype(np.int32)).cuda()
    sigma = (rng.integers(0, 2, d) * 2 - 1).astype(np.int8)
    pools = [M.Pool(d, hkv, hkv, 8, 8, sigma, max_batch=B) for _ in range(2)]
    gen = torch.Generator(device="cuda:0").manual_seed(5)
    k, v = (torch.randn((8 * 16, hkv, d), generator=gen, device="cuda:0", dtype=torch.bfloat16) for _ in range(2))
    for p in pools:
        p.append(k, v, torch.arange(8 * 16, dtype=torch.int32, device="cuda:0"))
        p.demote(torch.arange(8, dtype=torch.int32, device="cuda:0"), torch.arange(8, dtype=torch.int32, device="cuda:0"))
    q = torch.randn((B, hkv, d), generator=gen, device="cuda:0", dtype=torch.bfloat16)
    bt = torch.randint(0, 8, (B, 4), generator=gen, device="cuda:0", dtype=torch.int32)
    tags = torch.full((B, 4), M.TAG_RECENT, dtype=torch.uint8, device="cuda:0")
    tags[:, 0] = torch.where(lens >= 16, M.TAG_STALE, M.TAG_RECENT).to(torch.uint8)
    results = []
    for width in (4, wide):
        bts, tgs = torch.full((B, width), -1, dtype=torch.int32, device="cuda:0"), torch.zeros((B, width), dtype=torch.uint8, device="cuda:0")
        bts[:, :4], tgs[:, :4] = bt, tags
        new = lambda: (torch.full((B, hkv, d), float("nan"), device="cuda:0"), torch.full((B, hkv), float("nan"), device="cuda:0"))
        one, static, scored, layers = new(), new(), new(), (new(), new())
        pools[0].decode_attention(q, bts, tgs, lens, 0.1, out=one[0], lse=one[1])
        M.decode_attention_static(pools[0], q, bts, tgs, lens, 0.1, out=static[0], lse=static[1])
        mass = pools[0].decode_attention_scored(q, bts, tgs, lens, 0.1, out=scored[0], lse=scored[1])[2]
        M.decode_attention_layers(pools, [q] * 2, [bts] * 2, [tgs] * 2, lens, 0.1, [x[0] for x in layers], [x[1] for x in layers])
        torch.cuda.synchronize()
        assert all(p.status() == M.OK for p in pools) and not any(_tickets(p).any() for p in pools)
        assert not mass[:, :, 4:].any()
        results.append([*one, *static, *scored, *layers[0], *layers[1], mass[:, :, :4].clone()])
        del mass, bts, tgs
    for narrow, got in zip(*results):
        same = torch.isneginf(narrow)
        assert torch.equal(same, torch.isneginf(got))
        # sums of at most 64 terms in fp32, cut over other blocks: a few 2^-24 of the largest term
        assert (got[~same] - narrow[~same]).abs().max() < 1e-5
