"""GPU parity at the sizes where a kernel's tiles, ranges and dispatch rules have their edges."""
import numpy as np
import pytest
import torch

import cf_synth as syn
import oracle
import paper_2609_27085_b200 as cf
from harness import GpuScenario, compare, run_and_check, to_dev_bf16, to_host_bits
from test_gpu_parity import _spike_run

pytestmark = pytest.mark.gpu


def small(seed, Hq, Hkv, D, prefix, qlens, NB=2048):
    return syn.scenario_from_lengths("e", syn.Geometry(Hq, Hkv, D, 16, NB), seed, prefix, qlens)


@pytest.mark.parametrize("Hq,Hkv,D", [(16, 2, 128), (16, 2, 64), (8, 2, 128), (4, 2, 64), (3, 3, 128)])
@pytest.mark.parametrize("window,split", [(0, 0), (0, 3), (70, 0), (1500, 3)])
def test_chunks_around_the_packed_q_tile(Hq, Hkv, D, window, split):
    """A q tile of the prefill kernel holds 128 / G tokens x G heads, an item two of them, a planner block 128 tokens:
    chunk lengths one short of, at and one past each of these, on prefixes that are not tile- or page-aligned."""
    G = Hq // Hkv
    t = 128 // G
    qlen = sorted({2, t - 1, t, t + 1, 2 * t - 1, 2 * t, 2 * t + 1, 127, 128, 129, 128 + t, 128 + 2 * t + 1} - {0, 1})
    prefix = [(211 * i * i + 7 * i) % 2500 for i in range(len(qlen))]
    run_and_check(small(61, Hq, Hkv, D, prefix, [qlen]), window=window, sinks=None if window == 0 else np.linspace(-2, 2, Hq, dtype=np.float32),
                  debug={cf.CF_DEBUG_PREFILL_SPLIT: split} if split else None)


@pytest.mark.parametrize("Hq,Hkv,D", [(16, 2, 64), (8, 2, 128), (2, 2, 128)])
@pytest.mark.parametrize("window", [1, 31, 32, 33, 95, 129])
def test_windows_around_the_skipped_column_chunks(Hq, Hkv, D, window):
    """The softmax leaves out chunks of 32 columns that no row of a warp sees: windows one short of, at and one past a
    chunk, on chunks of every length class, so that leading, middle and trailing chunks of a tile are dead."""
    run_and_check(small(67, Hq, Hkv, D, [0, 5, 1000, 1023, 313, 64], [[150, 40, 129, 33, 300, 1]]), window=window)


@pytest.mark.parametrize("Hq,Hkv,D", [(16, 2, 64), (8, 2, 128), (2, 2, 128)])
def test_causal_edges_around_the_masked_column_chunks(Hq, Hkv, D):
    """The causal mask is applied to the 32-column chunks that it crosses: prefixes one short of, at and one past a
    chunk's and a tile's edge."""
    run_and_check(small(68, Hq, Hkv, D, [0, 30, 31, 32, 33, 95, 127, 128], [[1, 33, 40, 2, 64, 130, 3, 31]]))


@pytest.mark.parametrize("Hq,Hkv,D,fp8", [(2, 2, 64, False), (8, 2, 128, False), (24, 24, 64, False), (32, 8, 128, True), (24, 24, 128, True)])
@pytest.mark.parametrize("n_seqs", [1, 2, 31, 32, 33, 65, 1030])
def test_append_at_the_edges_of_the_row_search(Hq, Hkv, D, fp8, n_seqs):
    """The append's search splits the sequences 32 ways per step and moves a row in rounds of 32 x 8 loads: sequence counts
    around powers of 32, empty sequences at the front, between and at the end, rows of less and more than one round
    (24 heads).  Bit-exact whole-pool compare (inside run_and_check) and attention on top."""
    rng = np.random.default_rng(n_seqs)
    qlen = rng.choice([0, 0, 1, 1, 2, 5], size=n_seqs)
    qlen[rng.integers(n_seqs)] = 3
    prefix = rng.integers(0, 40, size=n_seqs)
    scales = (rng.uniform(0.01, 0.03, Hkv).astype(np.float32), rng.uniform(0.01, 0.03, Hkv).astype(np.float32)) if fp8 else None
    run_and_check(small(71, Hq, Hkv, D, prefix, [qlen], NB=4096), fp8=scales)


@pytest.mark.parametrize("prefix,qlen", [
    ([900, 100, 2000, 50, 40], [650, 1, 1, 1, 1]),                    # one chunk, decode behind it
    ([3000, 100, 7, 0, 700, 512], [1, 1, 700, 0, 130, 2]),            # decode first; an empty sequence inside the prefill run
    ([0, 31, 16], [1500, 257, 900]),                                  # prefill alone, cut into parts
    ([5, 77, 300, 1000], [300, 1, 400, 1]),                           # four runs of alternating kind
    ([5, 77, 300, 1000, 9], [300, 1, 400, 1, 200]),                   # five runs: computed in one piece
])
@pytest.mark.parametrize("window", [0, 200])
def test_host_steps_in_parts(prefix, qlen, window):
    """A host-staged step with at least 4 MB of prefill rows is computed and read back in parts."""
    sc = small(73, 32, 8, 128, prefix, [qlen], NB=1024)
    b = sc.batches[0]
    g = GpuScenario(sc, window=window)
    pin = lambda x: torch.from_numpy(x.view(np.int16)).pin_memory()
    bt, qh, kh, vh = torch.from_numpy(b.block_table).cuda(), pin(b.q), pin(b.k_new), pin(b.v_new)
    k_ref, v_ref = sc.k_pool.copy(), sc.v_pool.copy()
    oracle.kv_append(k_ref, v_ref, b.k_new, b.v_new, b.block_table, b.context_len, b.query_len)
    rows = syn.tile_edge_rows(b)
    ref_o, _ = oracle.mixed_attention(b.q, k_ref, v_ref, b.block_table, b.context_len, b.query_len, rows=rows, window=window)
    for _ in range(4):                                                # more steps than staging sets
        oh = torch.full_like(qh, -1).pin_memory()
        cf.cf_mixed_step_host(g.ctx, g.desc, qh, kh, vh, g.k, g.v, bt, b.max_blocks, b.context_len, b.query_len, oh)
        cf.cf_host_steps_flush(g.ctx)
    torch.cuda.synchronize()
    assert cf.cf_get_async_status(g.ctx) == cf.CF_OK
    compare(oh.numpy().view(np.uint16), None, ref_o, None, rows=rows)
    kg, vg = g.pools_host()
    assert np.array_equal(kg, k_ref) and np.array_equal(vg, v_ref)
    g.close()


def test_host_steps_without_a_flush_in_between():
    """A step whose kernels outweigh its copies goes in parts when it comes first after a flush and in one piece when it
    follows another: both against the oracle, three in flight, the same bits."""
    sc = small(74, 32, 8, 128, [40000, 3000], [[600, 1]], NB=3072)
    b = sc.batches[0]
    g = GpuScenario(sc)
    pin = lambda x: torch.from_numpy(x.view(np.int16)).pin_memory()
    bt, qh, kh, vh = torch.from_numpy(b.block_table).cuda(), pin(b.q), pin(b.k_new), pin(b.v_new)
    k_ref, v_ref = sc.k_pool.copy(), sc.v_pool.copy()
    oracle.kv_append(k_ref, v_ref, b.k_new, b.v_new, b.block_table, b.context_len, b.query_len)
    rows = np.array([0, 31, 32, 127, 128, 599, 600])
    ref_o, _ = oracle.mixed_attention(b.q, k_ref, v_ref, b.block_table, b.context_len, b.query_len, rows=rows)
    outs = [torch.full_like(qh, -1).pin_memory() for _ in range(3)]
    for oh in outs:
        cf.cf_mixed_step_host(g.ctx, g.desc, qh, kh, vh, g.k, g.v, bt, b.max_blocks, b.context_len, b.query_len, oh)
    cf.cf_host_steps_flush(g.ctx)
    torch.cuda.synchronize()
    assert cf.cf_get_async_status(g.ctx) == cf.CF_OK
    for oh in outs:
        compare(oh.numpy().view(np.uint16), None, ref_o, None, rows=rows)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[1], outs[2])
    g.close()


@pytest.mark.parametrize("Hq,Hkv,D,fp8", [(16, 2, 64, False), (8, 2, 128, False), (2, 2, 128, False), (16, 2, 128, True)])
@pytest.mark.parametrize("lens", [
    [1], [16], [128], [129],                                          # one page, one shortest chunk, one page more
    [31 * 16, 32 * 16 + 1, 33 * 16],
    [2500, 1, 77, 4000, 640],                                         # chunks of 8 to 32 pages
    [193 * 16] * 3 + [192 * 16],                                      # around the longest chunk
    [300] * 150,                                                      # whole sequences fill the slots
])
def test_decode_chunk_lengths(Hq, Hkv, D, fp8, lens):
    """The decode chunk rule picks chunks of 8 to 192 pages or whole sequences: batches on both sides of its lines."""
    scales = (np.full(Hkv, 0.02, np.float32), np.full(Hkv, 0.015, np.float32)) if fp8 else None
    run_and_check(small(79, Hq, Hkv, D, [l - 1 for l in lens], [[1] * len(lens)], NB=4096), fp8=scales)


@pytest.mark.parametrize("Hq,Hkv,D,fp8,layout", [(16, 2, 64, False, "HND"), (8, 2, 128, False, "HND"), (16, 2, 128, True, "HND"),
                                                 (16, 2, 64, False, "NHD"), (8, 2, 128, False, "NHD")])
@pytest.mark.parametrize("window", [0, 83, 2500])
def test_decode_rings_of_every_depth(Hq, Hkv, D, fp8, layout, window):
    """A decode warp's ring holds three or four pages, and the warp keeps 32 block ids: every number of pages per warp around the
    ring's depth, past 32 and 64 ids, whole and cut last pages, a window's edge inside a page, both pool layouts.  The shortest
    chunk is set above every sequence's length, so that a warp has a quarter of its pages."""
    lens = [max(1, 16 * pages + extra) for pages in (0, 1, 2, 3, 4, 7, 8, 12, 13, 16, 19, 20, 24, 127, 130, 261) for extra in (0, 1, 15)]
    d = cf.make_desc(Hq, Hkv, D, 16, 4096, window_size=window)
    dec = cf.cf_plan_inspect(d, lens, [1] * len(lens), 512, decode_min_chunk_pages=272)[1]
    pages = np.ceil((dec[:, 3] - dec[:, 2]) / 16).astype(int)
    assert len(dec) == len(lens) and {1, 2, 3, 4, 5} <= set(pages.tolist()) and pages.max() == (262 if window == 0 else 7 if window == 83 else 158)
    scales = (np.full(Hkv, 0.02, np.float32), np.full(Hkv, 0.015, np.float32)) if fp8 else None
    run_and_check(small(83, Hq, Hkv, D, [l - 1 for l in lens], [[1] * len(lens)], NB=4096), fp8=scales, layout=layout, window=window,
                  debug={cf.CF_DEBUG_DECODE_MIN_CHUNK_PAGES: 272})


@pytest.mark.parametrize("Hq,Hkv,D,fp8", [(16, 2, 64, False), (8, 2, 128, False), (16, 2, 128, True)])
@pytest.mark.parametrize("window", [0, 83])
def test_decode_from_pools_of_every_layout(Hq, Hkv, D, fp8, window):
    """The decode kernels have an instantiation for pools whose (page, head) holds its tokens one behind the other, chosen when K and V
    both do, and one for all others: K and V each as [blocks, heads, tokens, D], [blocks, tokens, heads, D] and with a padded row give
    the same bits, decode and the pages of an fp8 cache that prefill reads (first and last pages cut, a window's edge inside a page)."""
    lens = [1, 15, 16, 17, 63, 64, 65, 129, 700, 1100, 2500, 400]
    scales = (np.full(Hkv, 0.02, np.float32), np.full(Hkv, 0.015, np.float32)) if fp8 else None
    qlen = [1] * 11 + [130]
    sc = small(89, Hq, Hkv, D, [l - q if q == 1 else l for l, q in zip(lens, qlen)], [qlen])
    b = sc.batches[0]
    g = GpuScenario(sc, window=window, fp8=scales)
    g.append(b)
    ref, ref_lse = g.attend(b)
    bt, q = torch.from_numpy(b.block_table).cuda(), to_dev_bf16(b.q)
    pad = 32

    def laid_out(pool, how):
        if how == "heads":
            return pool, (Hkv * 16 * D, 16 * D, D)
        rows = torch.zeros((pool.shape[0], 16, Hkv * D + (pad if how == "padded" else 0)), dtype=pool.dtype, device="cuda")
        rows[:, :, :Hkv * D] = pool.permute(0, 2, 1, 3).reshape(pool.shape[0], 16, Hkv * D)
        return rows, (16 * rows.shape[2], D, rows.shape[2])
    scale = dict(kv_dtype=cf.CF_KV_FP8_E4M3, k_scale=g.k_scale_dev, v_scale=g.v_scale_dev) if fp8 else {}
    for how_k, how_v in (("tokens", "tokens"), ("heads", "tokens"), ("tokens", "heads"), ("padded", "heads"), ("padded", "padded")):
        (k, ks), (v, vs) = laid_out(g.k, how_k), laid_out(g.v, how_v)
        d = cf.make_desc(Hq, Hkv, D, 16, sc.geom.num_blocks, k_strides=ks, v_strides=vs, window_size=window, **scale)
        out, lse = torch.full_like(q, float("nan")), torch.full((b.total_q, Hq), float("nan"), dtype=torch.float32, device="cuda")
        cf.cf_mixed_attention(g.ctx, d, q, k, v, bt, b.max_blocks, b.context_len, b.query_len, out, lse)
        torch.cuda.synchronize()
        assert cf.cf_get_async_status(g.ctx) == cf.CF_OK
        assert np.array_equal(to_host_bits(out), ref) and np.array_equal(lse.cpu().numpy(), ref_lse), (how_k, how_v)
    run_and_check(sc, window=window, fp8=scales)
    g.close()


@pytest.mark.parametrize("Hq,Hkv,D,members", [(2, 2, 128, 40), (8, 2, 128, 4), (8, 2, 128, 5), (8, 2, 128, 9), (8, 2, 128, 17),
                                              (16, 2, 64, 2), (16, 2, 64, 3), (16, 2, 64, 9), (4, 2, 128, 22), (4, 2, 64, 33)])
@pytest.mark.parametrize("pages", [16, 33, 129])
def test_shared_prefix_sets_of_every_width(Hq, Hkv, D, members, pages):
    """The warps of a shared-prefix CTA split the columns of a set (16 each) or its pages: sets that need one, two and
    four warps per page, sets cut at 64 columns and at 32 members, chunks with an odd number of pages."""
    own = [(37 * i * i) % 300 for i in range(members)]
    sc, sg, sl = syn.shared_prefix_scenario("sets", syn.Geometry(Hq, Hkv, D, 16, 2048), 80 + members, pages * 16, own, [1] * members,
                                            [0] * members)
    b = sc.batches[0]
    g = GpuScenario(sc)
    g.append(b)
    q = to_dev_bf16(b.q)
    out = torch.full_like(q, float("nan"))
    lse = torch.full((b.total_q, Hq), float("nan"), dtype=torch.float32, device="cuda")
    cf.cf_mixed_attention_shared(g.ctx, g.desc, q, g.k, g.v, torch.from_numpy(b.block_table).cuda(), b.max_blocks, b.context_len,
                                 b.query_len, sg, sl, out, lse)
    torch.cuda.synchronize()
    assert cf.cf_get_last_plan_counts(g.ctx)[6] == members
    k_ref, v_ref = g.pools_host()
    ref_o, ref_lse = oracle.mixed_attention(b.q, k_ref, v_ref, b.block_table, b.context_len, b.query_len)
    compare(to_host_bits(out), lse.cpu().numpy(), ref_o, ref_lse)
    g.close()


@pytest.mark.parametrize("Hq,Hkv,D", [(8, 2, 128), (16, 2, 64)])
@pytest.mark.parametrize("spike", [96.0, 192.0])
def test_spikes_around_the_chunk_that_is_handed_over_last(Hq, Hkv, D, spike):
    """The product P V starts on the first 96 columns of a tile before the exponentials of the last 32 exist, so whether
    the reference has to be raised is decided from those columns' scores: a towering key on both sides of that line."""
    Lq, P = 200, 1000
    cand = [128 * t + c for t in (1, 2, 5, P // 128) for c in (94, 95, 96, 97, 110, 111, 126, 127)]
    _spike_run(small(71, Hq, Hkv, D, [P], [[Lq]]), cand, [0, 1, 31, 32, 127, 128, Lq - 1], spike)


@pytest.mark.parametrize("Hq,Hkv,D,members", [(8, 2, 128, 0), (16, 2, 128, 0), (16, 2, 64, 0), (8, 2, 128, 4), (8, 2, 128, 9), (8, 2, 128, 16),
                                              (16, 2, 64, 8)])
def test_the_dominant_probability_is_not_rounded(Hq, Hkv, D, members):
    """One key, well behind the pages that a warp starts with, outweighs each of the others by 2^1 to 2^7.9 and alone has a
    value: relative to the running maximum its probability is 1, so the result differs from the oracle's by its own rounding to bf16
    (half a unit in the last place) and by what fp32 sums of 300 terms add (below 2^-13); a rounded probability adds up to 2^-8.  members > 0: the key is part of a shared prefix."""
    n = max(1, members)
    geom = syn.Geometry(Hq, Hkv, D, 16, 1024)
    if members:
        sc, sg, sl = syn.shared_prefix_scenario("dominant", geom, 91, 256, [5] * n, [1] * n, [0] * n)
    else:
        sc = small(91, Hq, Hkv, D, [127], [[1]], NB=1024)
    b = sc.batches[0]
    at = 150 if members else 70
    rng = np.random.default_rng(91)
    k, v = np.zeros_like(sc.k_pool), np.zeros_like(sc.v_pool)
    page, slot = int(b.block_table[0, at // 16]), at % 16
    k[page, :, slot, 0] = syn.f32_to_bf16_bits(np.float32(1.0))
    v[page, :, slot, :] = syn.f32_to_bf16_bits(rng.uniform(1.0, 2.0, (Hkv, D)).astype(np.float32))
    q = np.zeros_like(b.q)
    lead = np.linspace(1.0, 7.9, n * Hq).reshape(n, Hq)                    # log2 of the key's weight
    q[:, :, 0] = syn.f32_to_bf16_bits((lead * np.log(2.0) * np.sqrt(D)).astype(np.float32))
    g = GpuScenario(sc)
    g.k, g.v, qd = to_dev_bf16(k), to_dev_bf16(v), to_dev_bf16(q)
    out = torch.full_like(qd, float("nan"))
    args = (g.ctx, g.desc, qd, g.k, g.v, torch.from_numpy(b.block_table).cuda(), b.max_blocks, b.context_len, b.query_len)
    if members:
        cf.cf_mixed_attention_shared(*args, sg, sl, out)
        assert cf.cf_get_last_plan_counts(g.ctx)[6] == members
    else:
        cf.cf_mixed_attention(*args, out)
    torch.cuda.synchronize()
    ref, _ = oracle.mixed_attention(q, k, v, b.block_table, b.context_len, b.query_len)
    half_ulp = 2.0 ** (np.floor(np.log2(ref)) - 8)
    excess = (np.abs(syn.bf16_bits_to_f64(to_host_bits(out)) - ref) - half_ulp) / ref
    assert excess.max() <= 2.0 ** -13, excess.max()
    g.close()


@pytest.mark.parametrize("prefix,qlen", [
    ([3000, 4500, 6000], [45, 45, 45]),                               # few short chunks: KV ranges, planned anew without
    ([2500, 5000, 300, 1800, 40, 2900, 700], [1, 300, 1, 1, 1, 1, 1]),
    ([700] * 31, [1] * 31),                                           # a wave of short chunks, planned anew with long ones
    ([2600, 9, 1500, 2600, 1100, 2600], [1, 2, 1, 1, 600, 1]),
])
@pytest.mark.parametrize("window,fp8", [(0, False), (1000, False), (0, True)])
def test_a_small_fixed_workspace_is_planned_for(prefix, qlen, window, fp8):
    """A fixed workspace that the default plan's partials do not fit (1 MB, a quarter of it the ticket counters; an fp8 cache:
    the chunks' staging on top) is planned for with fewer chunks and KV ranges: whatever fits with 128-page decode chunks and
    uncut prefill items is served."""
    sc = small(95, 32, 8, 128, prefix, [qlen], NB=2048)
    pages = sum((p + q + 15) // 16 for p, q in zip(prefix, qlen) if q > 1)
    ctx = cf.cf_create(0, workspace_bytes=4096 + (2 * pages * 8 * 16 * 128 * 2 + 4 * len(prefix) * 1024 if fp8 else 0))
    scales = (np.full(8, 0.02, np.float32), np.full(8, 0.015, np.float32)) if fp8 else None
    run_and_check(sc, ctx=ctx, window=window, fp8=scales)
    cf.cf_destroy(ctx)


@pytest.mark.parametrize("members,served_shared", [(8, True), (20, True), (40, False)])
def test_a_small_fixed_workspace_and_shared_prefixes(members, served_shared):
    """The partials of eleven shared chunks per member outgrow 1 MB: the shared part goes in one chunk, or, where two slots per
    member are too many as well, the sequences are served one by one."""
    sc, sg, sl = syn.shared_prefix_scenario("ws", syn.Geometry(32, 8, 128, 16, 2048), 96, 2048, [7 * i for i in range(members)], [1] * members,
                                            [0] * members)
    b = sc.batches[0]
    ctx = cf.cf_create(0, workspace_bytes=4096)
    g = GpuScenario(sc, ctx=ctx)
    g.append(b)
    q = to_dev_bf16(b.q)
    out = torch.full_like(q, float("nan"))
    lse = torch.full((b.total_q, 32), float("nan"), dtype=torch.float32, device="cuda")
    cf.cf_mixed_attention_shared(ctx, g.desc, q, g.k, g.v, torch.from_numpy(b.block_table).cuda(), b.max_blocks, b.context_len,
                                 b.query_len, sg, sl, out, lse)
    torch.cuda.synchronize()
    assert (cf.cf_get_last_plan_counts(ctx)[6] > 0) == served_shared
    k_ref, v_ref = g.pools_host()
    ref_o, ref_lse = oracle.mixed_attention(b.q, k_ref, v_ref, b.block_table, b.context_len, b.query_len)
    compare(to_host_bits(out), lse.cpu().numpy(), ref_o, ref_lse)
    g.close()
    cf.cf_destroy(ctx)


def test_a_host_step_that_does_not_fit_is_refused_before_anything_is_enqueued():
    """fp8 cache: the staging of one chunk's context outgrows the fixed workspace.  The step is refused with the caches, out_host
    and the staging sets as they were, and the steps around it are served."""
    sc = small(97, 32, 8, 128, [0, 6000, 50], [[600, 40, 1]], NB=1024)
    b = sc.batches[0]
    scales = (np.full(8, 0.02, np.float32), np.full(8, 0.015, np.float32))
    ctx = cf.cf_create(0, workspace_bytes=8 << 20)                    # 38 staged pages (2.5 MB) fit, 378 (25 MB) do not
    g = GpuScenario(sc, ctx=ctx, fp8=scales)
    pin = lambda x: torch.from_numpy(x.view(np.int16)).pin_memory()
    qh, kh, vh, bt = pin(b.q), pin(b.k_new), pin(b.v_new), torch.from_numpy(b.block_table).cuda()
    fits = (np.array([600, 0, 51], np.int32), np.array([600, 0, 1], np.int32))
    idx = np.r_[0:600, 640]
    qs, ks, vs = (torch.from_numpy(x.view(np.int16)[idx].copy()).pin_memory() for x in (b.q, b.k_new, b.v_new))
    outs = []
    for step in range(7):                                             # the set of a refused step comes round again
        if step % 2:
            k0, v0 = g.pools_host()
            oh = torch.full_like(qh, 77).pin_memory()
            st = cf.cf_mixed_step_host(ctx, g.desc, qh, kh, vh, g.k, g.v, bt, b.max_blocks, b.context_len, b.query_len, oh, check=False)
            assert st == cf.CF_ERR_WORKSPACE
            cf.cf_host_steps_flush(ctx)
            torch.cuda.synchronize()
            k1, v1 = g.pools_host()
            assert bool((oh == 77).all()) and np.array_equal(k0, k1) and np.array_equal(v0, v1)
        else:
            outs.append(torch.full_like(qs, 77).pin_memory())
            cf.cf_mixed_step_host(ctx, g.desc, qs, ks, vs, g.k, g.v, bt, b.max_blocks, *fits, outs[-1])
    cf.cf_host_steps_flush(ctx)
    torch.cuda.synchronize()
    assert cf.cf_get_async_status(ctx) == cf.CF_OK
    kr, vr = g.pools_host()
    ref, _ = oracle.mixed_attention(b.q[idx], kr, vr, b.block_table, *fits, k_scale=g.k_scale, v_scale=g.v_scale)
    for o in outs:
        compare(o.numpy().view(np.uint16), None, ref, None)
    g.close()
    cf.cf_destroy(ctx)


@pytest.mark.parametrize("prefix,qlen,fp8", [
    ([40000, 3000], [600, 1], False),
    ([70, 9000, 40000, 3000, 500, 20000], [1, 1, 600, 300, 1, 1], False),
    ([40000, 36000, 100, 100], [300, 400, 0, 1], False),
    ([30000, 9000, 700], [600, 1, 1], True),
])
def test_a_host_step_does_not_depend_on_the_steps_before_it(prefix, qlen, fp8):
    """The first step after a flush goes in parts; those behind it, bound by their kernels, in one piece: the same bits, which are
    right."""
    sc = small(98, 32, 8, 128, prefix, [qlen], NB=5120)
    b = sc.batches[0]
    scales = (np.full(8, 0.02, np.float32), np.full(8, 0.015, np.float32)) if fp8 else None
    g = GpuScenario(sc, fp8=scales)
    pin = lambda x: torch.from_numpy(x.view(np.int16)).pin_memory()
    qh, kh, vh, bt = pin(b.q), pin(b.k_new), pin(b.v_new), torch.from_numpy(b.block_table).cuda()
    outs, kernels = [], []
    for _ in range(5):
        outs.append(torch.full_like(qh, -1).pin_memory())
        cf.cf_mixed_step_host(g.ctx, g.desc, qh, kh, vh, g.k, g.v, bt, b.max_blocks, b.context_len, b.query_len, outs[-1])
        kernels.append(cf.cf_get_last_plan_counts(g.ctx)[2])
    cf.cf_host_steps_flush(g.ctx)
    torch.cuda.synchronize()
    assert cf.cf_get_async_status(g.ctx) == cf.CF_OK
    assert kernels[0] == 0 < kernels[1]                               # the last call of a step in parts is its decode part
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    k_ref, v_ref = g.pools_host()
    rows = syn.tile_edge_rows(b)
    rows = np.unique(np.r_[rows[::9], rows[-3:], b.total_q - 1])
    variant = dict(k_scale=g.k_scale, v_scale=g.v_scale) if fp8 else {}
    ref, _ = oracle.mixed_attention(b.q, k_ref, v_ref, b.block_table, b.context_len, b.query_len, rows=rows, **variant)
    compare(outs[0].numpy().view(np.uint16), None, ref, None, rows=rows)
    g.close()
