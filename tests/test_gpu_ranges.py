"""Sizes at which the kernels' partitions and variants change: edges of tiles, remainders, the ends of their ranges."""
import numpy as np
import pytest
import torch

import locks_synth
import oracle
from common import t2np

pytestmark = pytest.mark.gpu


# Every problem's pages are sliced by its own length: requests of one token, a page less one, and one long request in the
# same row; 4, 16 and 3 heads per KV head; pages of several 16-token tiles that end inside a tile.  The bound is that of
# the attention tests: bf16 P and output.
@pytest.mark.parametrize("lens,Hq,Hkv,B,layout", [([16 * 450 + 3, 1, 33, 16 * 7], 8, 2, 16, "HND"), ([15, 16 * 700], 32, 2, 16, "NHD"),
                                                  ([5000, 16 * 400, 17] * 20, 6, 2, 16, "HND"), ([64 * 130 + 33, 64], 8, 2, 64, "HND"),
                                                  ([32 * 230, 49], 16, 1, 32, "NHD"), ([16 * 385], 4, 1, 16, "HND")])
def test_dense_attention_ragged_rows(lens, Hq, Hkv, B, layout):
    from gpu_util import GpuCase
    gc = GpuCase(locks_synth.Workload("ragged", lens, Hq=Hq, Hkv=Hkv, B=B, budget=16 * B, seed=len(lens) + Hq, layout=layout,
                                      tail_fill=float("nan")))
    out, lse = gc.gpu_attend()
    oout, olse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm)
    assert np.abs(out - oout).max() <= 2e-2
    assert np.abs(lse - olse).max() <= 1e-3 * max(1.0, np.abs(olse).max() / 10)
    assert gc.status() == 0


# The slices of a page list cover it once whatever their number: 128 of one long list, one page to a warp and fewer, lists that
# end one page into a slice or one before its end, and a row much longer than its requests.  The bound is that of P in bf16.
@pytest.mark.parametrize("lens,row,Hq,Hkv", [([16 * 8188 + 5], 0, 16, 1), ([16 * 901] * 4, 0, 32, 2), ([16 * 7], 0, 4, 4), ([16 * 297 + 1, 16 * 296], 0, 12, 1),
                                             ([16 * 149, 16 * 3, 16 * 148 + 1, 9] * 4, 3000, 8, 2), ([16 * 501], 0, 32, 8), ([16 * 60, 16 * 59 + 1] * 20, 500, 28, 4)])
def test_slices_of_dense_attention(lens, row, Hq, Hkv):
    import paper_2607_24555_b200 as locks
    from gpu_util import GpuCase
    from paper_2607_24555_b200.binding import KVView, make_config
    gc = GpuCase(locks_synth.Workload("slices", lens, Hq=Hq, Hkv=Hkv, budget=256, seed=Hq + len(lens), tail_fill=float("nan")))
    want, want_lse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm)
    if row:
        table = torch.zeros(len(lens), row, dtype=torch.int32, device="cuda:0")
        table[:, :gc.max_pages] = gc.case.block_table
        gc.ctx = locks.Context(make_config(Hq, Hkv, 8, "i4", "bf16", len(lens), row, 256))
        gc.kv = KVView(gc.case.k, gc.case.v, gc.case.strides, gc.case.num_blocks, table, gc.case.seq_lens)
    out, lse = gc.gpu_attend()
    assert np.abs(out - want).max() <= 2e-2
    assert np.abs(lse - want_lse).max() <= 1e-3 * max(1.0, np.abs(want_lse).max() / 10)
    assert gc.status() == 0


# A length beyond the table's row is reported, and the row is attended as if the length ended with it: the slices do not depend on
# pages that do not exist (and no loop walks them).
@pytest.mark.parametrize("dtype,B,rows,Hq,Hkv", [("bf16", 16, 64, 8, 2), ("bf16", 16, 61, 32, 2), ("bf16", 32, 40, 8, 2), ("f32", 16, 64, 8, 2), ("f32", 16, 500, 32, 8)])
def test_length_beyond_the_row(dtype, B, rows, Hq, Hkv):
    from gpu_util import GpuCase
    gc = GpuCase(locks_synth.Workload("long", [B * rows, B * 30], Hq=Hq, Hkv=Hkv, B=B, dtype=dtype, fmt="f32" if dtype == "f32" else "i4", budget=4 * B, seed=4))
    want, want_lse = gc.gpu_attend()
    assert gc.status() == 0
    for extra in (1, 5 * B, 10_000 * B):
        gc.case.seq_lens[0] = B * rows + extra
        out, lse = gc.gpu_attend()
        assert gc.status() == -6   # LOCKS_ERR_BAD_BLOCK
        assert np.array_equal(out, want) and np.array_equal(lse, want_lse)


# A length of zero or less attends nothing: zeros, and a log-sum-exp of minus infinity.
@pytest.mark.parametrize("dtype,B,Hq", [("bf16", 16, 8), ("bf16", 16, 32), ("bf16", 64, 8), ("f32", 16, 8)])
def test_length_of_nothing(dtype, B, Hq):
    from gpu_util import GpuCase
    gc = GpuCase(locks_synth.Workload("none", [B * 40, B * 30, B * 20], Hq=Hq, Hkv=2, B=B, dtype=dtype, fmt="f32" if dtype == "f32" else "i4", budget=4 * B, seed=4))
    want, want_lse = gc.gpu_attend()
    gc.case.seq_lens[0], gc.case.seq_lens[2] = 0, -1000 * B
    out, lse = gc.gpu_attend()
    assert not out[[0, 2]].any() and np.isneginf(lse[[0, 2]]).all()
    assert np.abs(out[1] - want[1]).max() <= 2e-2 and np.abs(lse[1] - want_lse[1]).max() <= 1e-5 * np.abs(want_lse[1]).max()
    assert gc.status() == 0


# Pages of 32 and 64 tokens: weights and sums in fp32.  Sums of 128 products and of a few thousand weighted values are off by
# 1e-6 of the result at most, a bf16 result's rounding boundary is that near to one value in a thousand; weights rounded to
# bf16 move a third of the results.
@pytest.mark.parametrize("B", [32, 64])
@pytest.mark.parametrize("lens,Hq,Hkv,qs,layout", [([40, 9.1], 8, 2, 1.0, "HND"), ([75.3], 32, 2, 2.0, "NHD"), ([30] * 6, 12, 4, 0.5, "HND"),
                                                   ([2.9, 21.4, 11.55], 5, 1, 1.0, "NHD"), ([8, 33.02] * 3, 3, 3, 1.0, "HND"), ([6] * 40, 8, 8, 1.0, "HND")])
def test_wide_page_attention_rounds_once(B, lens, Hq, Hkv, qs, layout):
    from gpu_util import GpuCase
    gc = GpuCase(locks_synth.Workload("wide", [int(n * B) for n in lens], Hq=Hq, Hkv=Hkv, B=B, budget=6 * B, seed=B + Hq, q_scale=qs,
                                      layout=layout, tail_fill=float("nan")))
    P = [-(-t // B) for t in gc.w.seq_lens]
    ids = np.stack([np.stack([np.pad(np.unique(np.linspace(0, p - 1, min(p, 6)).astype(np.int32)), (0, 6), constant_values=-1)[:6]] * Hkv) for p in P])
    cnt = (ids >= 0).sum(-1).astype(np.int32)
    for table in ((None, None), (ids, cnt)):
        out, lse = gc.gpu_attend(*table)
        oout, olse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm, *table)
        want = torch.from_numpy(oout).to(torch.bfloat16).double().numpy()
        assert (out != want).mean() <= 5e-3
        assert np.abs(lse - olse).max() <= 3e-6 * max(1.0, np.abs(olse).max() / 10)
    assert gc.status() == 0


def _page_keys(kind, B, rng):
    """[B, 128] keys: the workloads' structure, and pages whose Gram matrix has close, equal, few or no eigenvalues."""
    d = 128
    if kind == "identical":
        return np.tile(rng.standard_normal(d), (B, 1))
    if kind == "rank1":
        return rng.standard_normal(d) + np.outer(rng.standard_normal(B), rng.standard_normal(d))
    if kind == "orthogonal":     # B - 1 equal eigenvalues
        return np.eye(B, d) * 3.0
    if kind == "two_keys":       # one eigenvalue
        return np.where((np.arange(B) % 2 == 0)[:, None], rng.standard_normal(d), rng.standard_normal(d))
    if kind == "blocks":         # equal pairs of eigenvalues in decoupled blocks
        k = np.zeros((B, d))
        for i in range(B):
            k[i, (i // 4) * 8 + i % 4] = 2.0
        return k
    dirs = rng.standard_normal((6, d))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    k = 3.0 * rng.standard_normal(d) + (3.0 * rng.standard_normal((B, 6))) @ dirs + 0.1 * rng.standard_normal((B, d))
    return k * {"large": 2.0 ** 30, "small": 2.0 ** -50}.get(kind, 1.0)


# The page that a decode step has just filled, at every page size and rank.  What is compared does not depend on the
# basis inside a (near-)degenerate eigenspace: the singular values, the residual of the rank-r summary, orthonormal
# rows.  The fp32 Gram matrix is off by 2^-24 x sqrt(128 B) of its largest eigenvalue (1e-5 at B = 64).
@pytest.mark.parametrize("B", [16, 32, 64])
@pytest.mark.parametrize("kind", ["structured", "identical", "rank1", "orthogonal", "two_keys", "blocks", "large", "small"])
def test_step_build_of_a_filled_page(B, kind):
    from gpu_util import GpuCase
    for r in (1, 2, 8, 16):
        w = locks_synth.Workload("fill", [3 * B, 2 * B - 1, 5 * B], Hq=2, Hkv=2, B=B, dtype="f32", fmt="f32", rank=r, budget=2 * B, seed=B + r)
        gc = GpuCase(w)
        rng = np.random.default_rng(B * 100 + r)
        keys = {}
        for b in (0, 2):
            blk = int(gc.case.block_table[b, w.seq_lens[b] // B - 1])
            for h in range(2):
                keys[b, h] = (blk, _page_keys(kind, B, rng).astype(np.float32))
                gc.case.k[blk, h] = torch.from_numpy(keys[b, h][1])
        summ = gc.ctx.new_summaries(gc.case.num_blocks)
        out = torch.empty(w.n, w.Hq, w.d, device="cuda:0")
        gc.ctx.locks_build_summaries(gc.kv, w.n, summ, torch.zeros(3, dtype=torch.int32, device="cuda:0"),
                                     torch.tensor([2, 1, 4], dtype=torch.int32, device="cuda:0"))   # all but the filled pages
        gc.ctx.locks_decode_step(gc.case.q, None, None, gc.kv, summ, w.n, out)
        assert gc.status() == 0
        got = summ.cpu().numpy()
        for (b, h), (blk, k) in keys.items():
            mu, V, Cc = oracle.unpack(gc.fmt, r, got[blk, h], B, w.d)
            D = k.astype(np.float64) - k.astype(np.float64).mean(0)
            sv = np.linalg.svd(D, compute_uv=False)[:r]
            top = max(float(sv[0]), 1e-30)
            keep = (sv ** 2 > 4e-6 * sv[0] ** 2) & (sv > 1e-4 * np.linalg.norm(k))   # clearly above the zero-mode thresholds
            assert np.abs(mu - k.astype(np.float64).mean(0)).max() <= 1e-6 * max(np.abs(k).max(), 1e-30)
            assert np.abs(np.linalg.norm(Cc, axis=0) - sv)[keep].max(initial=0.0) <= 1e-4 * top, (r, b, h)
            n = int(keep.sum())
            assert np.abs(V[:n] @ V[:n].T - np.eye(n)).max(initial=0.0) <= 2e-4, (r, b, h)
            res = np.linalg.norm(D - Cc @ V)
            best = np.sqrt(max((D ** 2).sum() - (sv[:n] ** 2).sum(), 0.0))
            assert res <= best + 2e-3 * top, (r, b, h, res, best)
        del gc


# The bulk kernel of bf16 keys and int4 summaries: ranges that start and end inside a warp's eight pages, every rank, both
# cache layouts, pages whose modes vanish.  Bytes against the oracle's fp64 build: a code differs where the value sits at a
# rounding boundary or two magnitudes of a mode are within fp32 of each other (the sign); 2e-4 of the bytes on random pages.
@pytest.mark.parametrize("rank", [2, 4, 8])
@pytest.mark.parametrize("layout", ["HND", "NHD"])
def test_bulk_build_partial_warps_and_degenerate_pages(rank, layout):
    from gpu_util import GpuCase
    w = locks_synth.Workload("bulk", [16 * 37, 16 * 8 + 5, 16 * 25 + 15], Hq=6, Hkv=3, rank=rank, budget=64, seed=rank, layout=layout)
    gc = GpuCase(w)
    rng = np.random.default_rng(rank)
    view = gc.case.k if layout == "HND" else gc.case.k.transpose(1, 2)
    flat = {}
    for i, kind in enumerate(["identical", "rank1", "orthogonal", "two_keys", "blocks"]):
        blk = int(gc.case.block_table[0, 3 + i])
        flat[blk] = kind
        view[blk] = torch.from_numpy(np.stack([_page_keys(kind, 16, rng) for _ in range(3)])).to(view)
    from common import oracle_cache
    gc.cache = oracle_cache(gc.case)
    want = gc.oracle_summaries()
    summ = gc.ctx.new_summaries(gc.case.num_blocks)
    begin, end = torch.tensor([1, 0, 17], dtype=torch.int32, device="cuda:0"), torch.tensor([30, 8, 25], dtype=torch.int32, device="cuda:0")
    gc.ctx.locks_build_summaries(gc.kv, w.n, summ, begin, end)
    assert gc.status() == 0
    got = summ.cpu().numpy()
    total = differ = 0
    for b, (lo, hi) in enumerate(zip([1, 0, 17], [30, 8, 25])):
        for page in range(-(-w.seq_lens[b] // 16)):
            blk = int(gc.case.block_table[b, page])
            if not lo <= page < hi:
                assert not got[blk].any(), (b, page)
                continue
            if blk in flat:   # bases inside an eigenspace are arbitrary: what counts is the reconstruction
                for h in range(3):
                    g = oracle.unpack(gc.fmt, rank, got[blk, h], 16, w.d)
                    o = oracle.unpack(gc.fmt, rank, want[blk, h], 16, w.d)
                    k = view[blk, h].double().cpu().numpy()
                    D = k - k.mean(0)
                    worse = np.linalg.norm(D - g[2] @ g[1]) - np.linalg.norm(D - o[2] @ o[1])
                    assert worse <= 0.1 * max(np.linalg.norm(D), 1e-6), (flat[blk], worse)   # half an int4 step: 1/14 per entry
                    assert np.abs(g[0] - o[0]).max() <= np.abs(o[0]).max() / 100
                continue
            total += got[blk].size
            differ += int((got[blk] != want[blk]).sum())
    assert differ <= 2e-3 * total, (differ, total)


# Modes just above the threshold below which they are dropped (an eigenvalue of 1e-6 of the largest): they are kept, so they have to
# have converged.  Their eigenvalues are known to 3 % in fp32, and the lengths of their basis vectors to half of that.
@pytest.mark.parametrize("B", [16, 32, 64])
@pytest.mark.parametrize("r", [2, 4, 8])
def test_step_build_of_weak_modes(B, r):
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    n, gen = 512, torch.Generator().manual_seed(B + r)
    U = torch.linalg.qr(torch.cat([torch.ones(n, B, 1), torch.randn(n, B, 7, generator=gen)], 2).double())[0][:, :, 1:]   # centred
    V = torch.linalg.qr(torch.randn(n, 128, 7, generator=gen).double())[0]
    sv = (torch.rand(n, 7, generator=gen) * 1.5e-6 + 1.3e-6).sqrt()
    sv[:, 0] = 1.0
    keys = ((U * sv[:, None]) @ V.transpose(1, 2)).float().cuda()[:, None].contiguous()
    ctx = locks.Context(make_config(2, 1, r, "f32", "f32", n, 3, 2 * B, B=B))
    kv = KVView(keys, keys, (B * 128, B * 128, 128), n, torch.arange(n, dtype=torch.int32, device="cuda:0")[:, None].repeat(1, 3).contiguous(),
                torch.full((n,), B, dtype=torch.int32, device="cuda:0"))
    summ, q = ctx.new_summaries(n), torch.zeros(n, 2, 128, device="cuda:0")
    ctx.locks_decode_step(q, None, None, kv, summ, n, torch.empty_like(q))
    assert ctx.locks_poll_status() == 0
    basis = summ.view(n, -1).view(torch.float32)[:, 128:128 + 128 * r].reshape(n, r, 128).norm(dim=2)
    assert bool((basis[:, 0] - 1).abs().max() < 5e-5)   # the fp32 Gram matrix: 2^-24 x sqrt(128 B) x 4 deviations at B = 64
    assert bool(((basis == 0) | ((basis - 1).abs() < 0.1)).all()), basis.max()


# The quantised formats of the page that a decode step fills, the last row being the step's own token.  The buffer is full of ones
# before: a byte that is not written shows.  Ordinary pages against the oracle's fp64 build: everything within one code of it once a
# mode's sign is settled, and one byte in a thousand different (bf16 entries: one in 200).  Pages whose bases are arbitrary inside an
# eigenspace: the reconstruction, as good as the oracle's but for half an int4 step (1/14 of an entry).
@pytest.mark.parametrize("B", [16, 32, 64])
@pytest.mark.parametrize("fmt", ["i4", "i8", "bf16"])
def test_step_build_of_a_filled_page_in_every_format(fmt, B):
    from common import oracle_cache
    from gpu_util import GpuCase
    kinds = [None] * 8 + ["identical", "rank1", "orthogonal", "two_keys", "blocks"]
    for r in (2, 4, 8):
        w = locks_synth.Workload("fill", [B * (2 + i % 3) for i in range(len(kinds))] + [2 * B + 5], Hq=4, Hkv=2, B=B, fmt=fmt, rank=r, budget=2 * B, seed=B + r)
        gc = GpuCase(w)
        rng = np.random.default_rng(B * 10 + r)
        kn, vn, qn = locks_synth.new_token(w, 0, device="cuda:0")
        blocks = [int(gc.case.block_table[b, -(-t // B) - 1]) for b, t in enumerate(w.seq_lens)]
        for b, kind in enumerate(kinds):
            page = None if kind is None else torch.from_numpy(np.stack([_page_keys(kind, B, rng) for _ in range(2)])).to(gc.case.k)
            if kind is not None:
                gc.case.k[blocks[b]] = page
            kn[b] = gc.case.k[blocks[b], :, B - 1] if page is None else page[:, B - 1]
            gc.case.k[blocks[b], :, B - 1] = 100.0   # the step writes this row
        gc.case.seq_lens -= 1
        summ = torch.full_like(gc.ctx.new_summaries(gc.case.num_blocks), 255)
        out = torch.empty(w.n, w.Hq, w.d, dtype=torch.bfloat16, device="cuda:0")
        gc.ctx.locks_decode_step(qn, kn, vn, gc.kv, summ, w.n, out)
        assert gc.status() == 0
        gc.cache = oracle_cache(gc.case)
        want, got = gc.oracle_summaries(), summ.cpu().numpy()
        assert np.array_equal(np.flatnonzero((got != 255).reshape(len(got), -1).any(1)), np.sort(blocks[:len(kinds)]))
        payload = oracle.summary_payload_bytes(gc.fmt, r, B, w.d)
        total = differ = 0
        for b, kind in enumerate(kinds):
            for h in range(2):
                g_blob, o_blob = got[blocks[b], h], want[blocks[b], h]
                assert not g_blob[payload:].any()
                g, o = oracle.unpack(gc.fmt, r, g_blob, B, w.d), oracle.unpack(gc.fmt, r, o_blob, B, w.d)
                step = {"i4": 1 / 7, "i8": 1 / 127, "bf16": 1 / 128}[fmt] * 1.01
                assert np.abs(g[0] - o[0]).max() <= np.abs(o[0]).max() / 126
                if kind is not None:
                    k = gc.case.k[blocks[b], h].double().cpu().numpy()
                    D = k - k.mean(0)
                    worse = np.linalg.norm(D - g[2] @ g[1]) - np.linalg.norm(D - o[2] @ o[1])
                    assert worse <= 0.1 * max(np.linalg.norm(D), 1e-6), (kind, worse)
                    continue
                flip = np.where((g[1] * o[1]).sum(1) < 0, -1.0, 1.0)
                assert (np.abs(g[1] * flip[:, None] - o[1]).max(1) <= step * np.abs(o[1]).max(1)).all()
                assert (np.abs(g[2] * flip - o[2]).max(1) <= 1.01 / 127 * np.abs(o[2]).max(1)).all()
                if (flip > 0).all():
                    total += payload
                    differ += int((g_blob[:payload] != o_blob[:payload]).sum())
        assert total > 0 and differ <= (5e-3 if fmt == "bf16" else 1e-3) * total, (differ, total)


def _bulk_bytes_by_key_type(keys, rank):
    """int4 summaries of pages [n, 16, 128] in one head: from bf16 keys (build_i4_group) and from the same values in fp32
    (build_kernel), which computes in the same order."""
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    n, got = len(keys), []
    for dt in (torch.bfloat16, torch.float32):
        ctx = locks.Context(make_config(2, 1, rank, "i4", "bf16" if dt == torch.bfloat16 else "f32", 1, n, 256))
        k = keys.to(dt).contiguous()
        kv = KVView(k, k, (2048, 2048, 128), n, torch.arange(n, dtype=torch.int32, device="cuda:0")[None].contiguous(),
                    torch.tensor([16 * n], dtype=torch.int32, device="cuda:0"))
        summ = ctx.new_summaries(n)
        ctx.locks_build_summaries(kv, 1, summ)
        assert ctx.locks_poll_status() == 0
        got.append(summ.view(n, -1))
    return got


# Sixteen keys with one large entry each and small ones beside it: 15 equal modes, and a 16th that is nothing but what the Gram
# matrix's diagonal lost in the sums, up to 3e-6 of the others.  It must not cost the page its basis.
@pytest.mark.parametrize("rank", [2, 4, 8])
def test_bulk_build_of_pages_with_equal_modes(rank):
    gen = torch.Generator().manual_seed(rank)
    pages = []
    for m in range(0, 128, 4):
        for e in range(-36, -16):
            big = 1.0 + m / 128.0
            k = 2.0 ** (e / 2) * big * (torch.randint(0, 2, (16, 128), generator=gen) * 2.0 - 1.0)
            k[torch.arange(16), torch.arange(16)] = big
            pages.append(k)
    bf, f32 = _bulk_bytes_by_key_type(torch.stack(pages).to(torch.bfloat16).cuda(), rank)
    at = 64 * rank + 16 * rank + 128 + 32   # the basis scales: fp16, one per mode
    assert bool((bf[:, at:at + 2 * rank].contiguous().view(torch.float16) > 0).all())
    assert torch.equal(bf, f32)


# Random pages, enough of them for values whose product with the inverse scale rounds to a tie (one in ten million): the bytes
# do not depend on the type that holds the keys.
@pytest.mark.parametrize("rank", [2, 4, 8])
def test_bulk_build_rounds_codes_alike(rank):
    gen = torch.Generator(device="cuda:0").manual_seed(rank)
    keys = 3.0 * torch.randn(100_000, 16, 128, generator=gen, device="cuda:0")
    bf, f32 = _bulk_bytes_by_key_type((keys + 2.0 * torch.randn(len(keys), 1, 128, generator=gen, device="cuda:0")).to(torch.bfloat16), rank)
    assert torch.equal(bf, f32), int((bf != f32).sum())


# The bulk build's ways to deal the pages out: by the table's rows (long rows in a pool that can fill them), one warp to a
# group of eight pages (many), two warps (few), and rounds of a grid that the pool bounds (eight layers, pages that share blocks).  Groups are the same eight pages
# each time, and the arithmetic does not depend on who works on them: the bytes are equal.
def test_bulk_build_is_dealt_out_in_several_ways():
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    dev, batch, hkv, rows = torch.device("cuda:0"), 40, 8, 264
    lens = [rows * 16 - 17 * (i % 3) for i in range(batch)]
    lens[3], lens[4], lens[33], lens[39] = 0, 15, 16 * 9 + 1, 16 * 8
    pages = [-(-t // 16) for t in lens]
    nb = 9000
    ctx = locks.Context(make_config(16, hkv, 8, "i4", "bf16", batch, rows, 256), device=dev)
    gen = torch.Generator(device=dev).manual_seed(5)
    k = torch.randn(nb, hkv, 16, 128, generator=gen, device=dev).to(torch.bfloat16)
    table = torch.randint(nb, (batch, rows), generator=gen, device=dev, dtype=torch.int32)   # pages may share a block
    seq = torch.tensor(lens, dtype=torch.int32, device=dev)
    kv = KVView(k, k, (hkv * 2048, 2048, 128), nb, table, seq)
    ones = torch.ones(batch, dtype=torch.int32, device=dev)
    builds = [ctx.new_summaries(nb) for _ in range(3)]
    ctx.locks_build_summaries(kv, batch, builds[0])
    ctx.locks_build_summaries(kv, batch, builds[1], 0 * ones, rows * ones)
    for at in range(0, rows, 64):
        ctx.locks_build_summaries(kv, batch, builds[2], at * ones, (at + 64) * ones)
    layers = [ctx.new_summaries(nb) for _ in range(8)]
    keep = ctx.locks_build_summaries_layers(kv, [k] * 8, layers, batch, 0 * ones, rows * ones)
    assert ctx.locks_poll_status() == 0 and keep
    host = table.cpu()
    built = torch.zeros(nb, dtype=torch.bool)
    for b, t in enumerate(lens):
        built[host[b, :t // 16].long()] = True
    assert torch.equal((builds[0].view(nb, -1) != 0).any(1).cpu(), built)
    once = np.bincount(np.concatenate([host[b, :t // 16].numpy() for b, t in enumerate(lens)]), minlength=nb) == 1
    once = torch.from_numpy(once).to(dev)   # a block in several pages is built beside other pages each time
    for other in builds[1:] + layers:
        assert torch.equal(builds[0][once], other[once])


# Short requests in long rows and a pool that could fill them: the same bytes as by page ranges, nothing outside, whatever takes them.
def test_bulk_build_of_short_requests_in_a_large_pool():
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    dev, hkv, row, nb = torch.device("cuda:0"), 8, 2176, 14_000
    lens = [2048, 16 * 7 + 15, 0, 16 * 8, 2100, 16 * 9, 1, 16 * 129]
    ctx = locks.Context(make_config(16, hkv, 8, "i4", "bf16", 8, row, 256), device=dev)
    gen = torch.Generator(device=dev).manual_seed(8)
    table = torch.full((8, row), -1, dtype=torch.int32, device=dev)   # slots past a request's pages are not looked at
    used = torch.randperm(nb, generator=gen, device=dev)[:sum(-(-t // 16) for t in lens)].to(torch.int32)
    at = 0
    for b, t in enumerate(lens):
        table[b, :-(-t // 16)] = used[at:at - (-t // 16)]
        at += -(-t // 16)
    k = torch.zeros(nb, hkv, 16, 128, dtype=torch.bfloat16, device=dev)
    k[used.long()] = torch.randn(len(used), hkv, 16, 128, generator=gen, device=dev).to(torch.bfloat16)
    kv = KVView(k, k, (hkv * 2048, 2048, 128), nb, table, torch.tensor(lens, dtype=torch.int32, device=dev))
    whole, ranges = ctx.new_summaries(nb), ctx.new_summaries(nb)
    ctx.locks_build_summaries(kv, 8, whole)
    ctx.locks_build_summaries(kv, 8, ranges, torch.zeros(8, dtype=torch.int32, device=dev), torch.full((8,), row, dtype=torch.int32, device=dev))
    assert ctx.locks_poll_status() == 0
    assert torch.equal(whole, ranges)
    assert int((whole.view(nb, -1) != 0).any(1).sum()) == sum(t // 16 for t in lens)


# The scan of int4 summaries at 32- and 64-token pages: every rank, one and two tiles of query heads, group sizes that fill
# neither, sequences that end inside a group of eight pages, more groups than warps (strides), extreme logits.
@pytest.mark.parametrize("B", [32, 64])
@pytest.mark.parametrize("lens,Hq,Hkv,rank,qs", [([40, 9, 17.5], 8, 2, 8, 1.0), ([33, 8.2], 32, 2, 8, 2.0), ([41], 12, 1, 4, 1.0),
                                                 ([25, 24, 18], 6, 3, 2, 1.0), ([900], 16, 1, 8, 4.0), ([60, 3], 2, 2, 4, 0.0)])
def test_wide_page_scan(B, lens, Hq, Hkv, rank, qs):
    from gpu_util import GpuCase, check_select_and_attend
    w = locks_synth.Workload("wide", [max(1, int(n * B)) for n in lens], Hq=Hq, Hkv=Hkv, B=B, rank=rank, budget=6 * B, seed=B + rank, q_scale=qs)
    gc = GpuCase(w)
    check_select_and_attend(gc, gc.oracle_summaries(), out_tol=2e-2)


# ... and its scores are no further from fp64 than those of the plain kernel in fp32 arithmetic, which scans the same summaries for
# fp32 queries of the same values.
@pytest.mark.parametrize("B", [32, 64])
@pytest.mark.parametrize("lens,Hq,Hkv,rank,qs", [([40, 30], 8, 2, 8, 1.0), ([200], 32, 2, 8, 2.0), ([60], 6, 3, 2, 1.0), ([60], 12, 1, 4, 1.0),
                                                 ([60], 8, 1, 8, 6.0), ([100], 28, 4, 4, 2.0)])
def test_wide_page_scan_is_as_accurate_as_fp32(B, lens, Hq, Hkv, rank, qs):
    import paper_2607_24555_b200 as locks
    from gpu_util import GpuCase, upload
    from paper_2607_24555_b200.binding import KVView, make_config
    w = locks_synth.Workload("wide", [n * B + 3 for n in lens], Hq=Hq, Hkv=Hkv, B=B, rank=rank, budget=6 * B, seed=B + rank, q_scale=qs)
    gc = GpuCase(w)
    summ = gc.oracle_summaries()
    want = oracle.page_logmass(gc.cache, t2np(gc.case.q), rank, gc.fmt, summ, float(np.float32(gc.sm)))
    fast = gc.gpu_select(upload(summ))[2]
    plain = GpuCase(w)
    plain.ctx = locks.Context(make_config(Hq, Hkv, rank, "i4", "f32", w.n, gc.max_pages, w.budget, B=B))
    k32 = gc.case.k.float()
    plain.kv = KVView(k32, k32, gc.case.strides, gc.case.num_blocks, gc.case.block_table, gc.case.seq_lens)
    slow = plain.gpu_select(upload(summ), gc.case.q.float())[2]
    off = [np.concatenate([np.abs(x[b, :, :n] - want[b, :, :n]).ravel() for b, n in enumerate(lens)]).mean() for x in (fast, slow)]
    assert off[0] <= off[1], off


# fp32 caches and summaries: one query head per KV head, fewer than four, more than four and not a multiple, sixteen; every
# rank of the fast scan and one beside them; last pages of 1, 8, 9 and 15 tokens, groups of eight pages that end early, splits
# without pages.  fp32 sums of 128 products: 1e-5 of outputs of a few units, scores 2e-7 of at most a hundred.
@pytest.mark.parametrize("rank", [2, 4, 8, 3])
@pytest.mark.parametrize("lens,Hq,Hkv,layout", [([16 * 40 + 1, 16 * 9 + 8], 2, 2, "HND"), ([16 * 77 + 9, 5, 16 * 17], 6, 2, "NHD"),
                                                ([16 * 30 + 15] * 3, 5, 1, "HND"), ([16 * 300, 16 * 8 + 1], 32, 2, "HND"),
                                                ([16 * 25 - 1] * 70, 8, 4, "HND")])
def test_fp32_scan_and_attention(lens, Hq, Hkv, layout, rank):
    from gpu_util import GpuCase, check_select_and_attend
    w = locks_synth.Workload("f32", lens, Hq=Hq, Hkv=Hkv, rank=rank, budget=16 * 7, dtype="f32", fmt="f32", seed=rank + Hq, layout=layout,
                             tail_fill=float("nan"))
    gc = GpuCase(w)
    check_select_and_attend(gc, gc.oracle_summaries(), out_tol=2e-5, mass_tol=1e-4)
    out, lse = gc.gpu_attend()
    oout, olse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm)
    assert np.abs(out - oout).max() <= 2e-5 and np.abs(lse - olse).max() <= 1e-4 * max(1.0, np.abs(olse).max() / 10)


# An infinite value makes an output infinite, not undefined, wherever in its tile the token sits: the last token of a page that is
# not full, of one that is, and one in the middle (bf16 caches of wide pages carry their weights in several parts).
@pytest.mark.parametrize("dtype,B", [("f32", 16), ("f32", 32), ("bf16", 32), ("bf16", 64)])
@pytest.mark.parametrize("Hq", [1, 4])
def test_infinite_values_stay_infinite(dtype, B, Hq):
    from gpu_util import GpuCase
    w = locks_synth.Workload("inf", [5 * B + 3, 4 * B - 1, 3 * B], Hq=Hq, Hkv=1, B=B, dtype=dtype, fmt="f32" if dtype == "f32" else "i4", budget=2 * B, seed=B)
    gc = GpuCase(w)
    want = torch.from_numpy(oracle.attend(gc.cache, t2np(gc.case.q), gc.sm)[0]).cuda()
    for b, (page, slot, dim, v) in enumerate([(5, 2, 5, "inf"), (3, B - 2, 70, "-inf"), (1, 9, 127, "inf")]):
        gc.case.v[int(gc.case.block_table[b, page]), 0, slot, dim] = float(v)
        want[b, :, dim] = float(v)
    out, _ = gc.gpu_attend()
    assert np.array_equal(np.isinf(out), torch.isinf(want).cpu().numpy()) and not np.isnan(out).any()
    assert np.array_equal(np.sign(out[np.isinf(out)]), torch.sign(want[torch.isinf(want)]).cpu().numpy())


# The K largest of up to 8192 keys in list order, ties to the earlier entry (exact: whole numbers against a sort).  Keys that
# leave the first histogram's threshold bin empty, full or crowded: all equal, two values, a crowd beside far outliers (a
# range of 32 bits), equal keys across the threshold, a smooth spread; as few as one winner, as many as there are entries.
@pytest.mark.parametrize("parts,kc", [(1, 1), (3, 1), (2, 30), (9, 126), (33, 126), (16, 510), (4, 2046), (8, 700)])
@pytest.mark.parametrize("kind", ["equal", "two", "outliers", "ties", "spread", "holes"])
def test_ranking_of_candidate_lists(parts, kc, kind):
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import make_config
    if parts * kc > 8192:
        pytest.skip("more entries than a ranking takes")
    rng = np.random.default_rng(parts * 31 + kc)
    ctx = locks.Context(make_config(2, 2, 8, "i4", "bf16", 2, 8000, (kc + 2) * 16))
    shape = (parts, 2, 2, kc)
    key = {"equal": np.full(shape, -3.25), "two": rng.choice([-1.0, -2.0], shape), "spread": -8.0 + 3.0 * rng.standard_normal(shape),
           "outliers": np.where(rng.random(shape) < 0.01, rng.choice([3e38, -3e38], shape), -5.0 + 1e-5 * rng.standard_normal(shape)),
           "ties": np.round(-6.0 + 2.0 * rng.standard_normal(shape), 1), "holes": -8.0 + 3.0 * rng.standard_normal(shape)}[kind].astype(np.float32)
    page = np.tile(np.arange(parts * kc, dtype=np.int32).reshape(parts, 1, 1, kc) * 7 + 1, (1, 2, 2, 1))
    if kind == "holes":
        page[rng.random(shape) < 0.9] = -1
    ids = torch.full((2, 2, kc), -7, dtype=torch.int32, device="cuda:0")
    cnt = torch.full((2, 2), -7, dtype=torch.int32, device="cuda:0")
    for _ in range(2):
        ctx.locks_merge_selection(torch.from_numpy(key).cuda(), torch.from_numpy(page).cuda(), 2, ids, cnt)
    ids, cnt = ids.cpu().numpy(), cnt.cpu().numpy()
    for b in range(2):
        for h in range(2):
            k, p = key[:, b, h].reshape(-1), page[:, b, h].reshape(-1)
            there = np.flatnonzero(p >= 0)
            best = np.sort(there[np.argsort(-k[there], kind="stable")[:kc]])
            assert cnt[b, h] == len(best)
            assert np.array_equal(ids[b, h, :len(best)], p[best])
            assert np.all(ids[b, h, len(best):] == -1)


# Selection in chunks whose lists together have fewer and more than 4096 entries (where the winners' pages are kept differs), with few
# and many winners.  All heads score a page alike, in steps that fp32 separates: the table is that of a stable sort.
@pytest.mark.parametrize("pages,Hq,Hkv,k", [(8448, 32, 2, 128), (20000, 16, 1, 300), (20000, 16, 1, 2000), (40000, 8, 1, 1000), (65792, 32, 2, 128), (65792, 32, 2, 3)])
def test_selection_from_chunk_lists(pages, Hq, Hkv, k):
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    rng = np.random.default_rng(pages + k)
    lens = [pages * 16 - 3, (pages - 777) * 16]
    ctx = locks.Context(make_config(Hq, Hkv, 8, "i4", "bf16", 2, pages, k * 16))
    dummy = torch.zeros(1, Hkv, 16, 128, dtype=torch.bfloat16, device="cuda:0")
    kv = KVView(dummy, dummy, (Hkv * 2048, 2048, 128), 1, torch.zeros(2, pages, dtype=torch.int32, device="cuda:0"),
                torch.tensor(lens, dtype=torch.int32, device="cuda:0"))
    score = (np.round(3.0 * rng.standard_normal((2, Hkv, 1, pages)) * 64) / 64).astype(np.float32)
    mass = torch.from_numpy(np.tile(score, (1, 1, Hq // Hkv, 1)).reshape(2, Hq, pages)).cuda()
    ids = torch.full((2, Hkv, k), -7, dtype=torch.int32, device="cuda:0")
    cnt = torch.full((2, Hkv), -7, dtype=torch.int32, device="cuda:0")
    for _ in range(2):
        ctx.locks_select_scored(torch.full((1, 2, Hq), -2.0, device="cuda:0"), kv, 2, ids, cnt, None, mass)
    assert ctx.locks_poll_status() == 0 and bool((cnt == k).all())
    for b, t in enumerate(lens):
        P = -(-t // 16)
        for h in range(Hkv):
            best = 1 + np.sort(np.argsort(-score[b, h, 0, 1:P - 1], kind="stable")[:k - 2])
            assert np.array_equal(ids[b, h].cpu().numpy(), np.concatenate([[0], best, [P - 1]]))


# A step whose build runs beside the scan counts the step's token itself, and the last of the request's page-heads and the selector
# stores the length.  Requests before, at and after a page boundary, and one without room for the token; KV heads that fill the
# build's CTAs (4, 2 or 1 page-heads) and that do not; three steps, so that what one step leaves behind shows in the next.
@pytest.mark.parametrize("Hkv", [1, 3, 4])
@pytest.mark.parametrize("B,dtype,fmt", [(16, "bf16", "i4"), (32, "bf16", "i4"), (64, "bf16", "i4"), (16, "f32", "f32"), (16, "bf16", "i8"), (32, "bf16", "bf16")])
def test_lengths_of_steps_whose_build_starts_at_once(B, dtype, fmt, Hkv):
    from gpu_util import GpuCase
    rows = 24
    w = locks_synth.Workload("lengths", [B * rows, B * 9 - 1, B * 9 - 2, B * 9, 1, B * 20 - 3], Hq=4 * Hkv, Hkv=Hkv, B=B, dtype=dtype,
                             fmt=fmt, rank=8, budget=4 * B, seed=B + Hkv)
    gc = GpuCase(w)
    want = gc.case.seq_lens.clone()
    summ = gc.gpu_build()
    before = summ.clone()
    out = torch.empty(w.n, w.Hq, w.d, dtype=gc.case.k.dtype, device="cuda:0")
    width = gc.case.block_table.shape[1] * B
    for step in range(3):
        kn, vn, qn = locks_synth.new_token(w, step, device="cuda:0")
        gc.ctx.locks_decode_step(qn, kn, vn, gc.kv, summ, w.n, out)
        torch.cuda.synchronize()
        want = torch.minimum(want + 1, torch.full_like(want, width))
        assert torch.equal(gc.case.seq_lens, want), step
        changed = (summ != before).reshape(len(summ), -1).any(1).nonzero().flatten().tolist()
        before = summ.clone()
        filled = [int(gc.case.block_table[b, int(t) // B - 1]) for b, t in enumerate(want.tolist()) if t % B == 0 and t > 0 and b > 0]
        assert set(filled) <= set(changed) <= set(filled) | {int(gc.case.block_table[0, rows - 1])}, step


# A request's last page may be an inner page of another one (a shared prompt of a whole number of pages).  The step writes its
# summary anew, but every score of the step is that of the old one, whichever is done first: the build (the plain scan of int8 bases with
# 16 heads takes ten times as long) or the scan.  The old summary here is another page's, so that the selections differ.
@pytest.mark.parametrize("B,fmt,dtype,rank,Hq,Hkv", [(16, "i4", "bf16", 8, 8, 2), (16, "i4", "bf16", 2, 32, 2), (16, "i8", "bf16", 2, 16, 1), (16, "bf16", "bf16", 4, 32, 2),
                                                     (16, "f32", "f32", 8, 8, 2), (32, "i4", "bf16", 8, 8, 2), (64, "i4", "bf16", 4, 12, 4), (32, "i8", "bf16", 8, 16, 1)])
def test_summary_of_a_shared_page_changes_after_the_scores(B, fmt, dtype, rank, Hq, Hkv):
    from gpu_util import GpuCase
    w = locks_synth.Workload("shared", [B * 41 + 3, B * 30, B * 37, B * 30], Hq=Hq, Hkv=Hkv, B=B, fmt=fmt, dtype=dtype, rank=rank, budget=6 * B, seed=B + rank)
    gc = GpuCase(w)
    gc.ctx.locks_set_scan_partition(1)
    table = gc.case.block_table
    table[1, :30] = table[0, :30]
    table[3, :30] = table[0, :30]
    shared = int(table[0, 29])
    own = [int(table[2, 36])]
    summ = gc.gpu_build()
    after = gc.gpu_select(summ)[0]
    best = int(table[0, int(np.nanargmax(gc.gpu_select(summ)[3][0, 0, 1:40])) + 1])
    assert best != shared
    old = summ.clone().reshape(gc.case.num_blocks, -1)
    old[shared] = old[best]
    want = gc.gpu_select(old.reshape(summ.shape))[:2]
    assert not np.array_equal(want[0][0], after[0])
    out = torch.empty(w.n, w.Hq, w.d, dtype=gc.case.k.dtype, device="cuda:0")
    results = []
    for _ in range(3):
        now = old.clone().reshape(summ.shape)
        ids = torch.full((w.n, Hkv, gc.k), -7, dtype=torch.int32, device="cuda:0")
        cnt = torch.full((w.n, Hkv), -7, dtype=torch.int32, device="cuda:0")
        gc.ctx.locks_decode_step(gc.case.q, None, None, gc.kv, now, w.n, out, ids, cnt)
        torch.cuda.synchronize()
        assert np.array_equal(ids.cpu().numpy(), want[0]) and np.array_equal(cnt.cpu().numpy(), want[1])
        results.append(now.reshape(old.shape))
        changed = (results[-1] != old).any(1).nonzero().flatten().tolist()
        assert shared in changed and set(changed) <= {shared, *own}
        assert torch.equal(results[-1], results[0])
    assert gc.status() == 0
    # the summary is a build's: nearly all bytes, or in fp32 the basis up to its signs
    built = summ.reshape(old.shape)[shared]
    if fmt == "f32":
        mu = [x.view(torch.float32).reshape(Hkv, -1)[:, :128] for x in (results[0][shared], built)]
        assert torch.allclose(mu[0], mu[1], rtol=0, atol=1e-5)   # fp32 sums of 16 keys of a few units
    else:
        assert (results[0][shared] != built).float().mean() <= 2e-2


# The splits of a problem merge through the shared memory of their cluster (16, 8, 4 or 2 CTAs, by the number of problems; the last
# case has one CTA each): slices of whole heads, of parts of heads and across heads, lists shorter than their row, an output buffer
# that is aligned to its elements only.  Tolerance: P and the result are rounded to bf16, each by at most 2^-9 of itself, and the
# weighted mean of |v| is no smaller than |out|.
@pytest.mark.parametrize("n,Hkv,G", [(1, 3, 5), (1, 2, 16), (3, 4, 1), (2, 4, 12), (5, 8, 7), (10, 4, 9), (5, 8, 16), (25, 4, 4), (25, 4, 3), (50, 4, 5), (64, 4, 8)])
def test_splits_merge_in_their_cluster(n, Hkv, G):
    from gpu_util import GpuCase
    w = locks_synth.Workload("merge", [900 + 7 * i % 60 if i % 5 else 100 + i for i in range(n)], Hq=G * Hkv, Hkv=Hkv, budget=768, seed=n + G)
    gc = GpuCase(w)
    ids, cnt, _, _ = gc.gpu_select(gc.gpu_build())
    want, want_lse = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm, ids, cnt)
    gc.cache.v &= 0x7FFF   # |v|, as bf16 bits
    bound = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm, ids, cnt)[0] * 2.0**-8 + 1e-5
    d_ids, d_cnt = torch.from_numpy(ids).cuda(), torch.from_numpy(cnt).cuda()
    for shift in (0, 1):
        out = torch.empty(w.n * w.Hq * w.d + 1, dtype=torch.bfloat16, device="cuda:0")[shift:][:w.n * w.Hq * w.d].view(w.n, w.Hq, w.d)
        lse = torch.empty(w.n, w.Hq, dtype=torch.float32, device="cuda:0")
        gc.ctx.locks_sparse_attend(gc.case.q, gc.kv, w.n, d_ids, d_cnt, out, lse)
        torch.cuda.synchronize()
        assert (np.abs(out.float().cpu().numpy() - want) <= bound).all() and np.abs(lse.cpu().numpy() - want_lse).max() <= 1e-3
    assert gc.status() == 0


# Infinite and undefined values pass the same merge: they reach the outputs of their dimension and no other.
@pytest.mark.parametrize("n,Hkv,G", [(1, 3, 5), (1, 2, 16), (5, 8, 7), (10, 4, 9), (25, 4, 4), (64, 4, 8)])
def test_infinite_values_pass_the_cluster_merge(n, Hkv, G):
    from gpu_util import GpuCase
    w = locks_synth.Workload("merge", [900 + 7 * i % 60 for i in range(n)], Hq=G * Hkv, Hkv=Hkv, budget=768, seed=n + G)
    gc = GpuCase(w)
    ids, cnt, _, _ = gc.gpu_select(gc.gpu_build())
    want = oracle.attend(gc.cache, t2np(gc.case.q), gc.sm, ids, cnt)[0]
    for b in range(n):
        for h in range(Hkv):
            for at, dim, v in ((0, 3, "inf"), (cnt[b, h] // 2, 64, "nan"), (cnt[b, h] - 1, 127, "-inf")):
                gc.case.v[int(gc.case.block_table[b, int(ids[b, h, at])]), h, 0, dim] = float(v)
                want[b, h * G:(h + 1) * G, dim] = float(v)
    out, lse = gc.gpu_attend(ids, cnt)
    assert np.array_equal(np.isnan(out), np.isnan(want)) and np.array_equal(np.isinf(out), np.isinf(want))
    assert np.array_equal(np.sign(out[np.isinf(out)]), np.sign(want[np.isinf(want)])) and np.isfinite(lse).all()
    there = np.isfinite(want)
    assert np.abs(out[there] - want[there]).max() <= 2e-2


# log Z from many partials, whole slices of them (32 of every warps-per-head x 32) and single ones at minus infinity, and scores at
# minus infinity for some of a group's heads.  The expected shares in fp64; scores and log Z of a few units, sums in fp32.
@pytest.mark.parametrize("Hq,Hkv", [(8, 2), (6, 1), (16, 2), (16, 1)])
@pytest.mark.parametrize("pages", [3000, 20000])
def test_log_shares_with_empty_slices_of_partials(pages, Hq, Hkv):
    import paper_2607_24555_b200 as locks
    from paper_2607_24555_b200.binding import KVView, make_config
    rng = np.random.default_rng(pages + Hq)
    G, k = Hq // Hkv, 64
    ctx = locks.Context(make_config(Hq, Hkv, 8, "i4", "bf16", 1, pages, k * 16))
    dummy = torch.zeros(1, Hkv, 16, 128, dtype=torch.bfloat16, device="cuda:0")
    kv = KVView(dummy, dummy, (Hkv * 2048, 2048, 128), 1, torch.zeros(1, pages, dtype=torch.int32, device="cuda:0"),
                torch.tensor([pages * 16 - 3], dtype=torch.int32, device="cuda:0"))
    mass = (3.0 * rng.standard_normal((1, Hq, pages))).astype(np.float32)
    mass[:, ::max(2, G), ::7] = -np.inf
    for nparts in (1, 33, 200, 360):
        parts = (2.0 * rng.standard_normal((nparts, 1, Hq))).astype(np.float32)
        parts[32:64] = -np.inf
        parts[96:128] = -np.inf
        parts[1::5] = -np.inf
        parts[:, 0, Hq - 1] = -np.inf
        parts[nparts - 1 if nparts < 33 else 20, 0, Hq - 1] = 0.5
        ids = torch.full((1, Hkv, k), -7, dtype=torch.int32, device="cuda:0")
        cnt = torch.full((1, Hkv), -7, dtype=torch.int32, device="cuda:0")
        share = torch.full((1, Hkv, pages), float("nan"), device="cuda:0")
        ctx.locks_select_scored(torch.from_numpy(parts).cuda(), kv, 1, ids, cnt, share, torch.from_numpy(mass).cuda())
        with np.errstate(divide="ignore"):
            logz = np.log(np.exp(parts.astype(np.float64)).sum(0))[0]
            want = np.log(np.exp(mass[0].astype(np.float64) - logz[:, None]).reshape(Hkv, G, pages).mean(1))
        got = share[0].cpu().numpy()[:, 1:-1]
        assert np.abs(got - want[:, 1:-1]).max() <= 1e-4
        for h in range(Hkv):
            best = 1 + np.sort(np.argsort(-got[h], kind="stable")[:k - 2])
            assert np.array_equal(ids[0, h].cpu().numpy(), np.concatenate([[0], best, [pages - 1]]))
