"""ckv_prefill: chunks of contiguous rows written into the paged cache with their summaries, against the cache image
and the summaries the prefill-time build produces from it."""
import numpy as np
import pytest
import torch

from paper_2609_26300_b200 import synth

from helpers import setup

pytestmark = pytest.mark.gpu

TOY = synth.CONFIGS[1]


def small(**kw):
    base = dict(batch=2, num_q_heads=8, num_kv_heads=2, ctx=16 * 40 + 11, budget_tokens=16 * 12, needles=0,
                outlier_dims=2, decode_steps=0, name="prefill")
    base.update(kw)
    return TOY.with_(**base)


def source_rows(w, dtype):
    """[batch][ctx][kv_heads][128] rows of the synthetic cache, as the projection layer would hand them over."""
    k = np.zeros((w.batch, w.ctx, w.num_kv_heads, 128), np.float32)
    v = np.zeros_like(k)
    lens = synth.seq_lens(w)
    for s in range(w.batch):
        for h in range(w.num_kv_heads):
            K, V = synth.unit_kv(w, s, h)
            k[s, :lens[s], h] = K[:lens[s]]
            v[s, :lens[s], h] = V[:lens[s]]
    return torch.from_numpy(k).to(dtype).cuda(), torch.from_numpy(v).to(dtype).cuda(), lens


@pytest.mark.parametrize("bs", [16, 32, 64])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("chunks", [(10 ** 6,), (37, 16, 1, 15, 200, 10 ** 6), (1, 1, 1, 62, 3, 10 ** 6)])
def test_chunked_prefill_equals_build(bs, dtype, chunks):
    w = small(block_size=bs, ctx_min=16 * 20 + 3)
    ref = setup(w, dtype)                                   # the cache image and the build over it
    ref.ckv.stats_build(ref.k_pool, ref.v_pool, ref.table, ref.lens, ref.max_len)
    want = [t.clone() for t in ref.ckv.export_stats(w.batch)]
    d = setup(w, dtype)
    d.k_pool.fill_(float("nan")); d.v_pool.fill_(float("nan"))
    k_src, v_src, lens = source_rows(w, dtype)
    cur = torch.zeros(w.batch, dtype=torch.int32, device="cuda")
    done = np.zeros(w.batch, np.int64)
    for c in chunks:
        new = np.minimum(c, lens - done).astype(np.int32)
        if new.max() == 0:
            break
        # every sequence's chunk starts at row 0 of its slice of the source buffer
        ks = torch.zeros(w.batch, int(new.max()), w.num_kv_heads, 128, dtype=dtype, device="cuda")
        vs = torch.zeros_like(ks)
        for s in range(w.batch):
            ks[s, :new[s]] = k_src[s, done[s]:done[s] + new[s]]
            vs[s, :new[s]] = v_src[s, done[s]:done[s] + new[s]]
        d.ckv.prefill(d.k_pool, d.v_pool, d.table, cur, ks, vs, torch.from_numpy(new).cuda(), int(new.max()))
        done += new
        torch.cuda.synchronize()
        assert np.array_equal(cur.cpu().numpy(), done)
    assert d.ckv.read_status() == 0
    assert np.array_equal(done, lens)
    got = d.ckv.export_stats(w.batch)
    for s in range(w.batch):
        n = int(lens[s]); x = -(-n // bs)
        for t in range(0, n, 16):                           # cache rows, bit for bit
            pg = int(d.table[s, t // 16]); m = min(16, n - t)
            assert torch.equal(d.k_pool[pg, :, :m], ref.k_pool[pg, :, :m])
            assert torch.equal(d.v_pool[pg, :, :m], ref.v_pool[pg, :, :m])
        for g, r in zip(got, want):                         # summaries, bit for bit
            assert torch.equal(g[s, :, :x], r[s, :, :x])


def test_prefill_then_decode_steps_and_capacity():
    w = small(ctx=16 * 30 + 5, decode_steps=4)
    ref = setup(w)
    ref.ckv.stats_build(ref.k_pool, ref.v_pool, ref.table, ref.lens, ref.max_len)
    d = setup(w)
    k_src, v_src, lens = source_rows(w, torch.bfloat16)
    cur = torch.zeros(w.batch, dtype=torch.int32, device="cuda")
    d.ckv.prefill(d.k_pool, d.v_pool, d.table, cur, k_src, v_src, torch.from_numpy(lens).cuda(), int(lens.max()))
    q = torch.from_numpy(synth.queries(w, 0)).bfloat16().cuda()
    a = d.ckv.decode(q, d.k_pool, d.v_pool, d.table, cur, d.max_len, w.budget_tokens)
    b = ref.ckv.decode(q, ref.k_pool, ref.v_pool, ref.table, ref.lens, ref.max_len, w.budget_tokens)
    torch.cuda.synchronize()
    assert torch.equal(a[0], b[0]) and torch.equal(a[2], b[2]) and torch.equal(a[3], b[3])
    # more tokens than the page table can hold: the excess is dropped and flagged
    cap = d.ckv.layout.max_blocks_per_seq * w.block_size
    room = cap - int(cur.max())
    extra = torch.full((w.batch,), room + 7, dtype=torch.int32, device="cuda")
    ks = torch.zeros(w.batch, room + 7, w.num_kv_heads, 128, dtype=torch.bfloat16, device="cuda")
    before = cur.clone()
    d.ckv.prefill(d.k_pool, d.v_pool, d.table, cur, ks, ks, extra, room + 7)
    torch.cuda.synchronize()
    assert d.ckv.read_status() & 2
    assert torch.all(cur == torch.minimum(before + room + 7, torch.full_like(cur, cap)))


@pytest.mark.parametrize("batch,tokens,bs", [(1, 2048, 16), (2, 8200, 16), (3, 20011, 16), (2, 16390, 32)])   # 1, 2 and more blocks per warp
def test_prefill_and_build_with_several_blocks_per_warp(batch, tokens, bs):
    """Launches of one and of several waves: both give the plain means (fp32 sums of 16 to 64 bf16 rows in [-6, 6] err by less
    than 64 * 6 * 2^-24, the stored pairs by 2^-18 of 6), and the prefill the same bits as the build."""
    from paper_2609_26300_b200 import binding
    hkv, pages = 8, -(-tokens // 64) * 4
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    k_src, v_src = (torch.randn(batch, tokens, hkv, 128, generator=gen, device="cuda").clamp(-6, 6).bfloat16() for _ in range(2))
    table = torch.randperm(batch * pages, generator=gen, device="cuda").int().view(batch, pages).contiguous()
    pools = [torch.zeros(batch * pages, hkv, 16, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    ckv = binding.CompKV(32, hkv, batch, pages * 16 // bs, batch * pages, block_size=bs)
    lens = torch.zeros(batch, dtype=torch.int32, device="cuda")
    new = torch.full_like(lens, tokens)
    new[-1] -= 5
    ckv.prefill(pools[0], pools[1], table, lens, k_src, v_src, new, tokens)
    got = [t.clone() for t in ckv.export_stats()]
    ckv.stats_build(pools[0], pools[1], table, lens, tokens)
    again = ckv.export_stats()
    torch.cuda.synchronize()
    assert torch.equal(lens, new) and ckv.read_status() == 0
    for s in range(batch):
        full, x = int(lens[s]) // bs, -(-int(lens[s]) // bs)
        for a, b in zip(got, again):
            assert torch.equal(a[s, :, :x], b[s, :, :x])
        want = k_src[s, :full * bs].view(full, bs, hkv, 128).double().mean(1).transpose(0, 1)
        assert float((got[0][s, :, :full].double() - want).abs().max()) <= 64 * 6 * 2.0 ** -24 + 6 * 2.0 ** -18


@pytest.mark.parametrize("bs", [16, 32, 64])
@pytest.mark.parametrize("bound", [4096, 16384, 65536])
def test_build_of_a_long_sequence_among_short_ones(bs, bound):
    """The blocks a warp takes follow from the host's bound and the batch: every sequence's summaries are those of a build
    of that sequence alone, whatever the bound."""
    w = small(batch=9, block_size=bs, ctx=16 * 90 + 11, ctx_min=5)
    d = setup(w)
    d.ckv.stats_build(d.k_pool, d.v_pool, d.table, d.lens, d.max_len)
    ref = [t.clone() for t in d.ckv.export_stats(w.batch)]
    blocks = bound // bs
    from paper_2609_26300_b200 import binding
    table = torch.full((w.batch, bound // 16), -1, dtype=torch.int32, device="cuda")
    table[:, :d.table.shape[1]] = d.table
    ckv = binding.CompKV(8, 2, w.batch, blocks, d.k_pool.shape[0], block_size=bs)
    ckv.stats_build(d.k_pool, d.v_pool, table, d.lens, bound)
    got = ckv.export_stats(w.batch)
    one = binding.CompKV(8, 2, 1, blocks, d.k_pool.shape[0], block_size=bs)
    for s in range(w.batch):
        n = -(-int(d.lens[s]) // bs)
        one.stats_build(d.k_pool, d.v_pool, table[s:s + 1].contiguous(), d.lens[s:s + 1].contiguous(), int(d.lens[s]))
        for x, y, z in zip(ref, got, one.export_stats(1)):
            assert torch.equal(x[s, :, :n], y[s, :, :n]) and torch.equal(x[s, :, :n], z[0, :, :n])
    assert d.ckv.read_status() == 0 and ckv.read_status() == 0 and one.read_status() == 0
