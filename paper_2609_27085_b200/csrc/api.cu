// C ABI of the library: context, plan upload and the launch sequence.
// See include/crossflow_attn.h for the contract of every entry point.
#include <cuda.h>

#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/crossflow_attn.h"
#include "kernels.h"
#include "plan.h"

namespace cf {

static constexpr int kRing = 4;                         // plan slots in flight
static constexpr size_t kDefaultWorkspace = 64u << 20;  // split-K partials
static constexpr size_t kDefaultPlanBytes = 1u << 20;
// The first kCounterBytes of a split-K workspace hold the fused-combine ticket counters of the decode kernel
// (one per first partial slot of a split sequence and KV head): zeroed when the buffer is allocated, put back
// to zero by the kernel.  A batch with more counters than fit uses the separate combine kernel.
static constexpr size_t kCounterBytes = 256u << 10;

struct TimedCall {
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    bool ran[3] = {false, false, false};
};

// Device staging of one host-buffer step (cf_mixed_step_host): inputs copied in on one copy stream,
// result copied out on another, so that the copies of neighbouring steps overlap the kernels.
static constexpr int kHostStages = 3;
static constexpr int kHostParts = 8;       // parts of a step whose results are read back one by one
struct HostStage {
    uint8_t* dev = nullptr;
    size_t bytes = 0;
    cudaEvent_t h2d_done = nullptr, h2d_kv_done = nullptr, compute_done = nullptr, d2h_done = nullptr;
    cudaEvent_t part_done[kHostParts] = {};
    bool used = false;
};

// TMA tensor maps of the prefill kernel, kept per (base address, geometry): a serving loop passes the same
// pools and activation buffer call after call (one set per layer), and encoding three maps costs a few
// microseconds of host time per launch.
struct PoolMapEntry {
    const void* base = nullptr;
    int D = 0, num_blocks = 0, Hkv = 0;
    int64_t sb = 0, sh = 0, st = 0;
    uint64_t stamp = 0;
    CUtensorMap map;
};
struct QMapEntry {
    const void* base = nullptr;
    int D = 0, rows = 0, Hq = 0, heads = 0;
    uint64_t stamp = 0;
    CUtensorMap map;
};
// q maps: a host-staged step has one base address per prefill part and staging set (with 8 entries the nine of three parts over three
// sets were encoded anew in every step)
static constexpr int kPoolMaps = 32, kQMaps = 8 + kHostStages * kHostParts;

struct PlanSlot {
    uint8_t* host = nullptr;   // pinned
    uint8_t* dev = nullptr;
    cudaEvent_t done = nullptr;
    cudaEvent_t uploaded = nullptr;   // host-staged steps: the plan copy runs on the input copy stream
    bool used = false;
};

}  // namespace cf

struct cf_ctx {
    int device = 0;
    int num_sms = 0;
    cf::PlanConfig cfg;
    cf::PlanSlot slots[cf::kRing];
    size_t plan_bytes = 0;
    int next_slot = 0;
    float* workspace = nullptr;
    size_t workspace_bytes = 0;
    bool workspace_fixed = false;
    uint32_t* queue_dev = nullptr;    // ticket and exit counter of the persistent prefill CTAs of unplanned calls: zero between calls (the last CTA resets them)
    uint32_t* err_dev = nullptr;      // [0] device-side findings (bit 0: a wait expired, bit 1: block id outside the pool); [1] scratch counter of cf_validate_block_table
    bool fused_combine = true; // split-K merge inside the decode kernel (CF_DEBUG_SEPARATE_COMBINE: the separate combine kernel)
    bool use_pairs = false;    // CF_DEBUG_PREFILL_PAIRS: chunked prefill on pairs of SMs where the geometry allows it (measured slower
                               // than one CTA per item, see prefill_tc2.cu; kept as a tested alternative)
    std::atomic<int> live_plans{0};
    // concurrent execution of the prefill kernel beside decode + combine
    bool overlap = true;
    cudaStream_t upload_stream = nullptr;      // plan uploads of cf_kv_append / cf_mixed_attention
    uint64_t unflushed_steps = 0;   // host-staged steps since the last flush
    int spatial_sms = 0;       // SMs given to the first prefill grid in that mode (0 = three fifths)
    int spatial_sms_default = 0;   // CF_SPATIAL_SMS at cf_create: what cf_set_overlap(ctx, 1) goes back to
    // host-staged step
    cf::HostStage stage[cf::kHostStages];
    int next_stage = 0;
    cudaStream_t h2d_stream = nullptr, h2d_kv_stream = nullptr, d2h_stream = nullptr;
    // timing: one quad of events per timed call since the last cf_get_timing_sums
    bool timing = false;
    std::vector<cf::TimedCall> timed;
    size_t timed_used = 0;
    int launches = 0;
    // host time spent inside the entry points (benchmark instrumentation): nanoseconds and call counts
    int64_t host_ns_append = 0, host_ns_attention = 0, host_ns_planner = 0;
    int32_t host_calls_append = 0, host_calls_attention = 0;
    // tensor-map cache (least recently used entry is replaced)
    cf::PoolMapEntry pool_maps[cf::kPoolMaps];
    cf::QMapEntry q_maps[cf::kQMaps];
    uint64_t map_stamp = 0;
    int32_t last_counts[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // item counts of the plan the last cf_mixed_attention built
};

// A plan that lives on the device for as long as the caller wants: built once per scheduler iteration
// and used by every layer's append + attention calls (the lengths are the same for all layers).
struct cf_plan {
    cf_ctx* ctx = nullptr;
    cf_cache_desc desc;
    int32_t num_seqs = 0, max_blocks = 0;
    uint8_t* host = nullptr;       // pinned copy (source of the one upload)
    uint8_t* dev = nullptr;
    float* part = nullptr;         // this plan's own split-K partials
    int n_part_slots = 0, n_pre_slots = 0;
    int n_stage_seqs = 0, n_stage_pages = 0, max_stage_pages = 0;
    cf::PlanRef ref;               // the lists in `dev`; behind them the lengths and the queue counters
    size_t off_len = 0, off_queue = 0, total = 0;
    int n_dec = 0, n_comb = 0, n_pre_tc = 0, n_pre_comb = 0, total_q = 0;
    bool pair = false;
    int front_sms = 0;          // spatial sequence: SMs of the first prefill grid (spatial_front_sms or cf_set_overlap)
};

namespace cf {

static int env_int(const char* name, int fallback)
{
    const char* v = std::getenv(name);
    if (!v || !*v) return fallback;
    char* end = nullptr;
    long x = std::strtol(v, &end, 10);
    return (end && *end == 0 && x > 0 && x < (1 << 20)) ? (int)x : fallback;
}

struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = (prev == dev) || cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard()
    {
        if (ok && prev >= 0) cudaSetDevice(prev);
    }
};

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

static cf_status ensure_plan_capacity(cf_ctx* c, size_t need)
{
    if (need <= c->plan_bytes) return CF_OK;
    size_t nb = c->plan_bytes ? c->plan_bytes : kDefaultPlanBytes;
    while (nb < need) nb *= 2;
    if (cudaDeviceSynchronize() != cudaSuccess) return CF_ERR_CUDA;
    for (int i = 0; i < kRing; ++i) {
        PlanSlot& s = c->slots[i];
        if (s.host) cudaFreeHost(s.host);
        if (s.dev) cudaFree(s.dev);
        s.host = s.dev = nullptr;
        s.used = false;
        if (cudaMallocHost((void**)&s.host, nb) != cudaSuccess) return CF_ERR_CUDA;
        if (cudaMalloc((void**)&s.dev, nb) != cudaSuccess) return CF_ERR_CUDA;
    }
    c->plan_bytes = nb;
    return CF_OK;
}

static cf_status ensure_workspace(cf_ctx* c, size_t need)
{
    if (need <= c->workspace_bytes) return CF_OK;
    if (c->workspace_fixed) return CF_ERR_WORKSPACE;
    if (cudaDeviceSynchronize() != cudaSuccess) return CF_ERR_CUDA;
    if (c->workspace) cudaFree(c->workspace);
    c->workspace = nullptr;
    c->workspace_bytes = 0;
    size_t nb = align_up(need + need / 4, 1u << 20);
    if (cudaMalloc((void**)&c->workspace, nb) != cudaSuccess) return CF_ERR_CUDA;
    // The ticket counters at its front start at zero.  cudaMemset runs on the legacy default stream, which is not
    // ordered against non-blocking streams: wait for it here, before any kernel of the caller's stream can count.
    if (cudaMemset(c->workspace, 0, kCounterBytes < nb ? kCounterBytes : nb) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
        return CF_ERR_CUDA;
    c->workspace_bytes = nb;
    return CF_OK;
}

// The lists of one call's plan, one behind the other (every offset a multiple of 16)
static size_t layout_of(const Plan& pl, size_t n_stage_seqs, PlanRef* r)
{
    size_t at = 0;
    auto list = [&](int32_t* off, size_t bytes) {
        *off = (int32_t)at;
        at = align_up(at + bytes, 16);
    };
    r->base = nullptr;
    list(&r->dec, sizeof(DecodeItem) * pl.decode.size());
    list(&r->comb, sizeof(CombineItem) * pl.combine.size());
    list(&r->sh, sizeof(SharedDecodeItem) * pl.shared_decode.size());
    list(&r->shm, sizeof(ShareMember) * pl.share_members.size());
    list(&r->pre_tc, sizeof(PrefillTcItem) * pl.prefill_tc.size());
    list(&r->pre_comb, sizeof(PrefillCombineItem) * pl.prefill_combine.size());
    list(&r->stage, sizeof(StageSeq) * n_stage_seqs);
    return at;
}
static int32_t shared_units(const Plan& pl, const cf_cache_desc* d)
{
    const int32_t per_unit = std::max(1, 16 / (d->num_q_heads / d->num_kv_heads));       // members whose heads fill the 16 columns of a warp
    int32_t n = 0;
    for (const SharedDecodeItem& it : pl.shared_decode) n += (it.n_members + per_unit - 1) / per_unit;
    return n;
}
static void write_plan(uint8_t* dst, const Plan& pl, const std::vector<StageSeq>& stage, const PlanRef& r)
{
    auto list = [&](int32_t off, const void* src, size_t bytes) {
        if (bytes) std::memcpy(dst + off, src, bytes);
    };
    list(r.dec, pl.decode.data(), sizeof(DecodeItem) * pl.decode.size());
    list(r.comb, pl.combine.data(), sizeof(CombineItem) * pl.combine.size());
    list(r.sh, pl.shared_decode.data(), sizeof(SharedDecodeItem) * pl.shared_decode.size());
    list(r.shm, pl.share_members.data(), sizeof(ShareMember) * pl.share_members.size());
    list(r.pre_tc, pl.prefill_tc.data(), sizeof(PrefillTcItem) * pl.prefill_tc.size());
    list(r.pre_comb, pl.prefill_combine.data(), sizeof(PrefillCombineItem) * pl.prefill_combine.size());
    list(r.stage, stage.data(), sizeof(StageSeq) * stage.size());
}

// Takes the next pinned slot (waits for its last use) ...
static cf_status next_slot(cf_ctx* c, size_t bytes, PlanSlot** out)
{
    cf_status st = ensure_plan_capacity(c, bytes);
    if (st != CF_OK) return st;
    PlanSlot& s = c->slots[c->next_slot];
    c->next_slot = (c->next_slot + 1) % kRing;
    if (s.used && cudaEventSynchronize(s.done) != cudaSuccess) return CF_ERR_CUDA;   // slot still in flight
    *out = &s;
    return CF_OK;
}
// ... and enqueues its upload.  The copy does not go on the caller's stream: there it would start only when that
// stream's earlier kernels are done (a few microseconds of copy-engine latency between kernels, every call) and, queued in
// the copy engine meanwhile, hold back copies enqueued after it.  It runs on a context-owned stream (a host-staged step:
// on its input copy stream) and the caller's stream waits for it through an event; the slot's device buffer is free by
// then (the host waited for the slot's last use).
static cf_status upload_slot(PlanSlot* s, size_t bytes, cudaStream_t copy_stream, cudaStream_t stream)
{
    if (cudaMemcpyAsync(s->dev, s->host, bytes, cudaMemcpyHostToDevice, copy_stream) != cudaSuccess) return CF_ERR_CUDA;
    if (cudaEventRecord(s->uploaded, copy_stream) != cudaSuccess || cudaStreamWaitEvent(stream, s->uploaded, 0) != cudaSuccess)
        return CF_ERR_CUDA;
    return CF_OK;
}

static cf_status finish_slot(PlanSlot* s, cudaStream_t stream)
{
    if (cudaEventRecord(s->done, stream) != cudaSuccess) return CF_ERR_CUDA;
    s->used = true;
    return CF_OK;
}

static int64_t now_ns()
{
    return std::chrono::duration_cast<std::chrono::nanoseconds>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

static const CUtensorMap* pool_map(cf_ctx* c, const void* base, const cf_cache_desc* d, int64_t sb, int64_t sh, int64_t st)
{
    PoolMapEntry* victim = &c->pool_maps[0];
    for (PoolMapEntry& e : c->pool_maps) {
        if (e.base == base && e.D == d->head_dim && e.num_blocks == d->num_blocks && e.Hkv == d->num_kv_heads && e.sb == sb &&
            e.sh == sh && e.st == st) {
            e.stamp = ++c->map_stamp;
            return &e.map;
        }
        if (e.stamp < victim->stamp) victim = &e;
    }
    if (!encode_pool_map(&victim->map, base, d->head_dim, d->num_blocks, d->num_kv_heads, sb, sh, st)) {
        victim->base = nullptr;
        return nullptr;
    }
    victim->base = base; victim->D = d->head_dim; victim->num_blocks = d->num_blocks; victim->Hkv = d->num_kv_heads;
    victim->sb = sb; victim->sh = sh; victim->st = st;
    victim->stamp = ++c->map_stamp;
    return &victim->map;
}

static const CUtensorMap* q_map(cf_ctx* c, const void* base, int D, int rows, int Hq, int heads)
{
    QMapEntry* victim = &c->q_maps[0];
    for (QMapEntry& e : c->q_maps) {
        if (e.base == base && e.D == D && e.rows == rows && e.Hq == Hq && e.heads == heads) {
            e.stamp = ++c->map_stamp;
            return &e.map;
        }
        if (e.stamp < victim->stamp) victim = &e;
    }
    if (!encode_q_map(&victim->map, base, D, rows, Hq, heads)) {
        victim->base = nullptr;
        return nullptr;
    }
    victim->base = base; victim->D = D; victim->rows = rows; victim->Hq = Hq; victim->heads = heads;
    victim->stamp = ++c->map_stamp;
    return &victim->map;
}

static float scale_log2_of(const cf_cache_desc* d)
{
    const float sc = d->softmax_scale > 0.f ? d->softmax_scale : 1.0f / std::sqrt((float)d->head_dim);
    return sc * 1.4426950408889634f;
}

}  // namespace cf

namespace cf {

struct PlanCounts {
    int n_dec = 0, n_comb = 0, n_shared = 0, n_pre_tc = 0, n_pre_comb = 0, total_q = 0;
    int n_stage_seqs = 0, n_stage_pages = 0, max_stage_pages = 0, num_seqs = 0;   // fp8 cache: pages to expand for the prefill chunks
    bool pair = false;          // the prefill items are pair items (two CTAs each)
    int front_sms = 0;          // spatial sequence: SMs of the first prefill grid, as the plan was balanced for
    int n_part_slots = 0;
};

// Split-K workspace: the ticket counters, decode partials [slot, Hq, D] + [slot, Hq, 2], then the compact
// partial rows of KV-split prefill items [row slot, D] + [row slot, 2].
// For an fp8 cache the workspace also holds the bf16 staging pools of the prefill chunks' pages (K and V,
// [stage page, Hkv, 16, D]) and the staging block table [S, max_blocks].
struct WsLayout {
    size_t dec_o = 0, dec_ml = 0, pre_o = 0, pre_ml = 0, stage_k = 0, stage_v = 0, stage_bt = 0, total = 0;
};
static WsLayout ws_layout(int n_part_slots, int n_pre_slots, int Hq, int D, int n_stage_pages = 0, int Hkv = 0, int64_t table_entries = 0)
{
    WsLayout w;
    w.dec_o = kCounterBytes;
    w.dec_ml = w.dec_o + align_up((size_t)n_part_slots * Hq * D * sizeof(float), 256);
    w.pre_o = w.dec_ml + align_up((size_t)n_part_slots * Hq * 2 * sizeof(float), 256);
    w.pre_ml = w.pre_o + align_up((size_t)n_pre_slots * D * sizeof(float), 256);
    w.stage_k = w.pre_ml + align_up((size_t)n_pre_slots * 2 * sizeof(float), 256);
    const size_t pool = n_stage_pages > 0 ? align_up((size_t)n_stage_pages * Hkv * 16 * D * 2, 1024) : 0;
    w.stage_v = w.stage_k + pool;
    w.stage_bt = w.stage_v + pool;
    w.total = w.stage_bt + (n_stage_pages > 0 ? align_up((size_t)table_entries * sizeof(int32_t), 256) : 0);
    return w;
}

// fp8 cache: which pages of which prefill sequences have to be expanded to bf16 for the prefill kernel (from the first
// page any row of the chunk can see - 0 without a sliding window - to the last page of the context)
static void stage_list(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len, int32_t S,
                       std::vector<StageSeq>* seqs, int* n_pages, int* max_pages)
{
    seqs->clear();
    *n_pages = 0;
    *max_pages = 0;
    if (d->kv_dtype != CF_KV_FP8_E4M3) return;
    for (int32_t s = 0; s < S; ++s) {
        if (query_len[s] <= 1) continue;
        const int32_t prefix = context_len[s] - query_len[s];
        const int32_t lo = d->window_size > 0 ? std::max(0, prefix - d->window_size + 1) : 0;
        StageSeq q;
        q.seq = s;
        q.page0 = lo / 16;
        q.n_pages = (context_len[s] + 15) / 16 - q.page0;
        q.stage_base = *n_pages;
        *n_pages += q.n_pages;
        *max_pages = std::max(*max_pages, q.n_pages);
        seqs->push_back(q);
    }
}

// Enqueues decode -> combine -> prefill for a plan that already sits in device memory
// (plan.base), or in host memory (hp), from where the launches carry it.  `queue`: the two counter words of the
// persistent prefill CTAs.  `serial`: not the spatial sequence, whatever cf_set_overlap says.
static cf_status launch_attention(cf_ctx* c, const cf_cache_desc* desc, const PlanCounts& n, const PlanRef& plan, const HostPlan& hp,
                                  uint32_t* queue, float* ws, const WsLayout& W, const void* q, const void* k_cache,
                                  const void* v_cache, const int32_t* block_table, int32_t max_blocks_per_seq, void* out,
                                  float* lse, cudaStream_t stream, bool serial, bool allow_timing)
{
    const int Hq = desc->num_q_heads, D = desc->head_dim;
    AttnParams p;
    p.q = (const __nv_bfloat16*)q;
    p.k_cache = (const __nv_bfloat16*)k_cache;
    p.v_cache = (const __nv_bfloat16*)v_cache;
    p.out = (__nv_bfloat16*)out;
    p.lse = lse;
    p.block_table = block_table;
    p.max_blocks = max_blocks_per_seq;
    p.num_blocks = desc->num_blocks;
    p.ks_block = desc->k_stride_block; p.ks_head = desc->k_stride_head; p.ks_token = desc->k_stride_token;
    p.vs_block = desc->v_stride_block; p.vs_head = desc->v_stride_head; p.vs_token = desc->v_stride_token;
    p.Hq = Hq; p.Hkv = desc->num_kv_heads; p.G = Hq / desc->num_kv_heads;
    p.scale_log2 = scale_log2_of(desc);
    p.window = desc->window_size;
    p.sinks = desc->sink_logits;
    const bool fp8 = desc->kv_dtype == CF_KV_FP8_E4M3;
    p.k_scale = fp8 ? desc->k_scale : nullptr;
    p.v_scale = fp8 ? desc->v_scale : nullptr;
    p.plan = plan;
    p.part_o = (float*)((uint8_t*)ws + W.dec_o);
    p.part_ml = (float*)((uint8_t*)ws + W.dec_ml);
    const bool fused_combine = c->fused_combine && n.n_shared == 0 && (size_t)n.n_part_slots * desc->num_kv_heads * sizeof(uint32_t) <= kCounterBytes;
    p.dec_chained = 0;
    p.dec_counters = fused_combine ? (uint32_t*)ws : nullptr;
    p.pre_part_o = (float*)((uint8_t*)ws + W.pre_o);
    p.pre_part_ml = (float*)((uint8_t*)ws + W.pre_ml);
    p.pre_queue = queue;
    p.err = c->err_dev;

    cudaError_t e = cudaSuccess;
    TimedCall* tc = nullptr;
    if (c->timing && allow_timing) {
        if (c->timed_used == c->timed.size()) {
            TimedCall fresh;
            bool ok = true;
            for (int i = 0; i < 4 && ok; ++i) ok = cudaEventCreate(&fresh.ev[i]) == cudaSuccess;
            if (!ok) return CF_ERR_CUDA;
            c->timed.push_back(fresh);
        }
        tc = &c->timed[c->timed_used++];
        tc->ran[0] = (n.n_dec > 0);
        tc->ran[1] = (n.n_comb > 0) && !fused_combine;
        tc->ran[2] = n.n_pre_tc > 0;
    }
    const bool has_prefill = n.n_pre_tc > 0;
    // the prefill kernels' view of the cache: the caller's pools, or (fp8 cache) the bf16 staging pools in the workspace
    AttnParams pp = p;
    cf_cache_desc pdesc = *desc;
    if (fp8 && has_prefill) {
        pp.k_cache = (const __nv_bfloat16*)((uint8_t*)ws + W.stage_k);
        pp.v_cache = (const __nv_bfloat16*)((uint8_t*)ws + W.stage_v);
        pp.block_table = (const int32_t*)((uint8_t*)ws + W.stage_bt);
        pp.num_blocks = n.n_stage_pages;
        pdesc.num_blocks = n.n_stage_pages;
        pdesc.k_stride_block = pdesc.v_stride_block = (int64_t)desc->num_kv_heads * 16 * D;
        pdesc.k_stride_head = pdesc.v_stride_head = 16 * D;
        pdesc.k_stride_token = pdesc.v_stride_token = D;
        pp.ks_block = pp.vs_block = pdesc.k_stride_block;
        pp.ks_head = pp.vs_head = pdesc.k_stride_head;
        pp.ks_token = pp.vs_token = pdesc.k_stride_token;
    }
    PrefillMaps maps;
    if (has_prefill) {
        const CUtensorMap* mq = q_map(c, q, D, n.total_q, Hq, n.pair ? 1 : p.G);
        const CUtensorMap* mk = pool_map(c, pp.k_cache, &pdesc, pdesc.k_stride_block, pdesc.k_stride_head, pdesc.k_stride_token);
        const CUtensorMap* mv = pool_map(c, pp.v_cache, &pdesc, pdesc.v_stride_block, pdesc.v_stride_head, pdesc.v_stride_token);
        if (!mq || !mk || !mv) return CF_ERR_CUDA;
        maps.q = *mq; maps.k = *mk; maps.v = *mv;
    }
    // fp8 cache: the pages of the prefill chunks are expanded first, on the caller's stream (the prefill kernel behind
    // it waits for the grid before it in the stream to complete before its first read)
    auto stage_pages = [&](cudaStream_t st) -> cudaError_t {
        if (!(fp8 && has_prefill)) return cudaSuccess;
        return launch_kv_dequant_gather(p, hp, n.n_stage_seqs, n.max_stage_pages,
                                        (__nv_bfloat16*)((uint8_t*)ws + W.stage_k), (__nv_bfloat16*)((uint8_t*)ws + W.stage_v),
                                        (int32_t*)((uint8_t*)ws + W.stage_bt), st);
    };
    auto decode_launch = [&](cudaStream_t st) -> cudaError_t {
        return fp8 ? launch_decode_fp8(p, hp, n.n_dec, st) : launch_decode_with_shared(p, hp, D, n.n_shared, n.n_dec, st);
    };
    int second_grid = 0;
    // Slots that take a prefill item: SMs, or pairs of SMs for pair items.  Grid sizes, the shared work queue and
    // the front / tail split below are counted in slots.
    const int per_slot = n.pair ? 2 : 1;
    const int sms = (c->num_sms > 0 ? c->num_sms : 148) / per_slot;
    const int pre_ctas = n.n_pre_tc < sms ? n.n_pre_tc : sms;      // persistent CTAs (pairs) of the serial sequence
    auto launch_prefill = [&](int n_slots, int queue_slots, int first_static, int ticket_base, int tail) {
        return n.pair ? launch_prefill_tc2(pp, maps, n.n_pre_tc, n_slots, queue_slots, first_static, ticket_base, tail, stream)
                      : launch_prefill_tc(pp, hp, maps, D, n.n_pre_tc, n_slots, queue_slots, first_static, ticket_base, tail, stream);
    };
    if (c->overlap && !serial && !tc && has_prefill && (n.n_dec > 0)) {
        // Spatial partition, three grids of one stream that run at the same time by programmatic launches.  `front`
        // persistent prefill CTAs (one per SM: a CTA takes an SM's whole shared memory) go first.  The decode grid is
        // allowed to start once every one of them holds its SM (they say so with griddepcontrol.launch_dependents) and
        // runs on the SMs left over.  A second prefill grid is allowed to start once the last decode CTA has, and draws
        // from the front grid's ticket counter, so the SMs that decode frees join the prefill.  The order in which the
        // grids reach the SMs decides the time: a decode grid that fills the machine first keeps the prefill CTAs, which
        // need an SM to themselves, out until its end.  Completion runs back along the chain (tail grid -> decode's extra
        // CTA -> front grid), so whatever follows in the stream sees all three done.  Against the same three grids on two
        // streams with a fork event, a join event and a stream memory operation that waited for the front CTAs, one pass
        // on a B200: chat mix 261 -> 246 us, its TP4 shard 96 -> 85 us, sliding-window layer 78 -> 71 us, agentic 930 ->
        // 917 us, tiny batch 43 -> 38 us (there the host's share of the saving).
        // The front grid's share comes from spatial_front_sms (or cf_set_overlap): decode keeps the SMs it needs to be
        // done by the time the prefill is.
        int front = (c->spatial_sms > 0 ? c->spatial_sms : n.front_sms > 0 ? n.front_sms : (c->num_sms * 3) / 5) / per_slot;
        if (front < 1) front = 1;
        if (front > sms) front = sms;
        if (front > n.n_pre_tc) front = n.n_pre_tc;
        int tail = n.n_pre_tc - front;
        if (tail > sms) tail = sms;
        second_grid = tail > 0;
        if (e == cudaSuccess) e = stage_pages(stream);
        if (e == cudaSuccess) e = launch_prefill(front, front + tail, 1, front, 0);
        p.dec_chained = 1;
        if (e == cudaSuccess) e = decode_launch(stream);
        if (e == cudaSuccess) e = launch_prefill(tail, front + tail, 0, front, 1);
        if (e == cudaSuccess) e = launch_combine(p, hp, D, fused_combine ? 0 : n.n_comb, stream);
        if (e == cudaSuccess) e = launch_prefill_combine(pp, hp, D, n.n_pre_comb, stream);
    } else {
        if (tc) cudaEventRecord(tc->ev[0], stream);
        if (e == cudaSuccess) e = decode_launch(stream);
        if (tc) cudaEventRecord(tc->ev[1], stream);
        if (e == cudaSuccess) e = launch_combine(p, hp, D, fused_combine ? 0 : n.n_comb, stream);
        if (tc) cudaEventRecord(tc->ev[2], stream);
        if (e == cudaSuccess) e = stage_pages(stream);
        if (e == cudaSuccess) e = launch_prefill(pre_ctas, pre_ctas, 1, pre_ctas, 0);
        if (e == cudaSuccess) e = launch_prefill_combine(pp, hp, D, n.n_pre_comb, stream);
        if (tc) cudaEventRecord(tc->ev[3], stream);
    }
    c->launches = (int)(n.n_dec > 0) + (int)(n.n_comb > 0 && !fused_combine) + (int)(n.n_pre_tc > 0) + (int)(n.n_pre_comb > 0) + second_grid;
    // a launch that failed half-way leaves tickets that no CTA will draw: the counters go back to zero behind the rest
    if (e != cudaSuccess && has_prefill) cudaMemsetAsync(queue, 0, 2 * sizeof(uint32_t), stream);
    return e == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}

}  // namespace cf

using namespace cf;

extern "C" {

const char* cf_status_string(cf_status s)
{
    switch (s) {
        case CF_OK: return "CF_OK";
        case CF_ERR_INVALID_ARG: return "CF_ERR_INVALID_ARG";
        case CF_ERR_UNSUPPORTED: return "CF_ERR_UNSUPPORTED";
        case CF_ERR_OUT_OF_RANGE: return "CF_ERR_OUT_OF_RANGE";
        case CF_ERR_WORKSPACE: return "CF_ERR_WORKSPACE";
        case CF_ERR_CUDA: return "CF_ERR_CUDA";
        case CF_ERR_TIMEOUT: return "CF_ERR_TIMEOUT";
        case CF_ERR_ARCH: return "CF_ERR_ARCH";
        case CF_ERR_BUSY: return "CF_ERR_BUSY";
    }
    return "CF_ERR_UNKNOWN";
}

cf_status cf_create(cf_ctx** out, int device, size_t workspace_bytes)
{
    if (!out) return CF_ERR_INVALID_ARG;
    *out = nullptr;
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) {
        cudaGetLastError();
        return count == 0 ? CF_ERR_CUDA : CF_ERR_INVALID_ARG;
    }
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return CF_ERR_CUDA;
    if (prop.major != 10) return CF_ERR_ARCH;
    DeviceGuard guard(device);
    if (!guard.ok) return CF_ERR_CUDA;
    cf_ctx* c = new (std::nothrow) cf_ctx();
    if (!c) return CF_ERR_CUDA;
    c->device = device;
    c->num_sms = prop.multiProcessorCount;
    c->cfg.num_sms = c->num_sms;
    {
        const char* v = std::getenv("CF_OVERLAP");          // spatial sequence unless CF_OVERLAP=0
        c->overlap = !(v && v[0] == '0' && v[1] == 0);
    }
    c->spatial_sms = c->spatial_sms_default = env_int("CF_SPATIAL_SMS", 0);
    bool ok = true;
    for (int i = 0; i < kRing && ok; ++i)
        ok = cudaEventCreateWithFlags(&c->slots[i].done, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&c->slots[i].uploaded, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && ensure_plan_capacity(c, kDefaultPlanBytes) == CF_OK;
    c->workspace_fixed = false;
    ok = ok && ensure_workspace(c, workspace_bytes ? workspace_bytes : kDefaultWorkspace) == CF_OK;
    c->workspace_fixed = workspace_bytes != 0;
    ok = ok && cudaStreamCreateWithFlags(&c->upload_stream, cudaStreamNonBlocking) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&c->h2d_stream, cudaStreamNonBlocking) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&c->h2d_kv_stream, cudaStreamNonBlocking) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&c->d2h_stream, cudaStreamNonBlocking) == cudaSuccess;
    for (int i = 0; i < kHostStages && ok; ++i) {
        ok = cudaEventCreateWithFlags(&c->stage[i].h2d_done, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&c->stage[i].h2d_kv_done, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&c->stage[i].compute_done, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&c->stage[i].d2h_done, cudaEventDisableTiming) == cudaSuccess;
        for (cudaEvent_t& ev : c->stage[i].part_done) ok = ok && cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess;
    }
    ok = ok && cudaMalloc((void**)&c->err_dev, 2 * sizeof(uint32_t)) == cudaSuccess;
    ok = ok && cudaMemset(c->err_dev, 0, 2 * sizeof(uint32_t)) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    ok = ok && cudaMalloc((void**)&c->queue_dev, 2 * sizeof(uint32_t)) == cudaSuccess;
    ok = ok && cudaMemset(c->queue_dev, 0, 2 * sizeof(uint32_t)) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        cf_destroy(c);
        return CF_ERR_CUDA;
    }
    *out = c;
    return CF_OK;
}

cf_status cf_destroy(cf_ctx* c)
{
    if (!c) return CF_ERR_INVALID_ARG;
    if (c->live_plans.load() > 0) return CF_ERR_BUSY;      // a plan holds a pointer to its context
    DeviceGuard guard(c->device);
    cudaDeviceSynchronize();
    for (int i = 0; i < kRing; ++i) {
        if (c->slots[i].host) cudaFreeHost(c->slots[i].host);
        if (c->slots[i].dev) cudaFree(c->slots[i].dev);
        if (c->slots[i].done) cudaEventDestroy(c->slots[i].done);
        if (c->slots[i].uploaded) cudaEventDestroy(c->slots[i].uploaded);
    }
    for (cf::TimedCall& tc : c->timed)
        for (int i = 0; i < 4; ++i)
            if (tc.ev[i]) cudaEventDestroy(tc.ev[i]);
    if (c->workspace) cudaFree(c->workspace);
    if (c->err_dev) cudaFree(c->err_dev);
    if (c->queue_dev) cudaFree(c->queue_dev);
    if (c->upload_stream) cudaStreamDestroy(c->upload_stream);
    for (int i = 0; i < kHostStages; ++i) {
        HostStage& hs = c->stage[i];
        if (hs.dev) cudaFree(hs.dev);
        if (hs.h2d_done) cudaEventDestroy(hs.h2d_done);
        if (hs.h2d_kv_done) cudaEventDestroy(hs.h2d_kv_done);
        if (hs.compute_done) cudaEventDestroy(hs.compute_done);
        if (hs.d2h_done) cudaEventDestroy(hs.d2h_done);
        for (cudaEvent_t ev : hs.part_done)
            if (ev) cudaEventDestroy(ev);
    }
    if (c->h2d_stream) cudaStreamDestroy(c->h2d_stream);
    if (c->h2d_kv_stream) cudaStreamDestroy(c->h2d_kv_stream);
    if (c->d2h_stream) cudaStreamDestroy(c->d2h_stream);
    delete c;
    return CF_OK;
}

}  // extern "C"

namespace cf {

static AppendParams append_params(cf_ctx* c, const cf_cache_desc* desc, void* k_cache, void* v_cache, const void* k_new, const void* v_new,
                                  const int32_t* block_table, int32_t max_blocks, int32_t num_seqs, int32_t total_rows)
{
    AppendParams p = {};
    p.k_cache = (__nv_bfloat16*)k_cache;
    p.v_cache = (__nv_bfloat16*)v_cache;
    p.k_new = (const __nv_bfloat16*)k_new;
    p.v_new = (const __nv_bfloat16*)v_new;
    p.block_table = block_table;
    p.max_blocks = max_blocks;
    p.ks_block = desc->k_stride_block; p.ks_head = desc->k_stride_head; p.ks_token = desc->k_stride_token;
    p.vs_block = desc->v_stride_block; p.vs_head = desc->v_stride_head; p.vs_token = desc->v_stride_token;
    p.Hkv = desc->num_kv_heads; p.D = desc->head_dim; p.num_seqs = num_seqs; p.total_rows = total_rows;
    p.num_blocks = desc->num_blocks; p.err = c->err_dev;
    p.k_scale = desc->kv_dtype == CF_KV_FP8_E4M3 ? desc->k_scale : nullptr;
    p.v_scale = desc->kv_dtype == CF_KV_FP8_E4M3 ? desc->v_scale : nullptr;
    return p;
}

// Enqueues the append of a validated batch (`pl`: q_start and total_q filled); a plan slot is uploaded on copy_stream.
static cf_status enqueue_append(cf_ctx* c, const cf_cache_desc* desc, Plan& pl, void* k_cache, void* v_cache, const void* k_new,
                                const void* v_new, const int32_t* block_table, int32_t max_blocks_per_seq, const int32_t* context_len,
                                const int32_t* query_len, int32_t num_seqs, cudaStream_t copy_stream, cudaStream_t stream)
{
    pl.prefix.clear();
    for (int32_t i = 0; i < num_seqs; ++i) pl.prefix.push_back(context_len[i] - query_len[i]);
    PlanSlot* slot = nullptr;
    AppendParams p = append_params(c, desc, k_cache, v_cache, k_new, v_new, block_table, max_blocks_per_seq, num_seqs, pl.total_q);
    if (num_seqs <= kAppendInlineSeqs) {
        p.host_q_start = pl.q_start.data();
        p.host_prefix = pl.prefix.data();
    } else {
        const size_t qs_bytes = sizeof(int32_t) * ((size_t)num_seqs + 1), pf_bytes = sizeof(int32_t) * (size_t)num_seqs;
        cf_status st = next_slot(c, qs_bytes + pf_bytes, &slot);
        if (st != CF_OK) return st;
        std::memcpy(slot->host, pl.q_start.data(), qs_bytes);
        std::memcpy(slot->host + qs_bytes, pl.prefix.data(), pf_bytes);
        st = upload_slot(slot, qs_bytes + pf_bytes, copy_stream, stream);
        if (st != CF_OK) return st;
        p.q_start = (const int32_t*)slot->dev;
        p.prefix = (const int32_t*)(slot->dev + qs_bytes);
    }
    const cudaError_t e = launch_kv_append(p, stream);
    const cf_status fs = slot ? finish_slot(slot, stream) : CF_OK;
    return e != cudaSuccess ? CF_ERR_CUDA : fs;
}

// One attention call, planned: everything that is decided from the lengths and can be refused, before anything is enqueued.
struct Unit {
    Plan pl;
    std::vector<StageSeq> stage;             // fp8 cache: pages to expand for the prefill chunks
    int n_stage_pages = 0, max_stage_pages = 0;
    int32_t num_seqs = 0, max_blocks = 0;
    WsLayout W;
    int front_sms = 0;
    bool serial = false;
};
static cf_status plan_unit(cf_ctx* c, const cf_cache_desc* desc, const int32_t* context_len, const int32_t* query_len, int32_t num_seqs,
                           int32_t max_blocks_per_seq, const int32_t* share_group, const int32_t* shared_len, bool serial, Unit* u)
{
    const int64_t t_in = now_ns();
    PlanConfig cfg = c->cfg;
    const int front_sms = !c->overlap || serial ? 0 : c->spatial_sms > 0 ? c->spatial_sms
                              : spatial_front_sms(desc, context_len, query_len, num_seqs, c->num_sms);
    cfg.prefill_sms_mixed = c->timing ? 0 : front_sms;
    cfg.prefill_pair = c->use_pairs && prefill_pair_supported(desc);
    Plan& pl = u->pl;
    cf_status st = build_plan(desc, context_len, query_len, num_seqs, max_blocks_per_seq, cfg, &pl, share_group, shared_len);
    if (st != CF_OK) return st;
    u->num_seqs = num_seqs;
    u->max_blocks = max_blocks_per_seq;
    u->serial = serial;
    if (!pl.prefill_tc.empty()) stage_list(desc, context_len, query_len, num_seqs, &u->stage, &u->n_stage_pages, &u->max_stage_pages);
    auto layout = [&](int n_part_slots, int n_pre_slots) {
        return ws_layout(n_part_slots, n_pre_slots, desc->num_q_heads, desc->head_dim, u->n_stage_pages, desc->num_kv_heads,
                         (int64_t)num_seqs * max_blocks_per_seq);
    };
    u->W = layout(pl.n_part_slots, pl.n_pre_slots);
    if (c->workspace_fixed && u->W.total > c->workspace_bytes) {
        // the batch is planned again for the partials that fit the caller's workspace (1 KB: the lists' alignment); one that
        // does not even fit without any is refused
        const int64_t left = (int64_t)c->workspace_bytes - (int64_t)layout(0, 0).total - 1024;
        cfg.part_bytes = left > 0 ? left : 0;
        st = build_plan(desc, context_len, query_len, num_seqs, max_blocks_per_seq, cfg, &pl, share_group, shared_len);
        if (st != CF_OK) return st;
        u->W = layout(pl.n_part_slots, pl.n_pre_slots);
        if (u->W.total > c->workspace_bytes) return CF_ERR_WORKSPACE;
    }
    u->front_sms = c->spatial_sms > 0 ? front_sms : pl.front_sms;
    c->host_ns_planner += now_ns() - t_in;
    return CF_OK;
}

// Enqueues a planned call.  ensure_workspace(c, u.W.total) has been called.
static cf_status enqueue_unit(cf_ctx* c, const cf_cache_desc* desc, const Unit& u, const void* q, const void* k_cache, const void* v_cache,
                              const int32_t* block_table, void* out, float* lse, cudaStream_t copy_stream, cudaStream_t stream)
{
    const Plan& pl = u.pl;
    // A small plan travels with the launches: up to kSmallPlanBytes with every kernel of the sequence, up to kMidPlanBytes
    // with the decode kernel when it is the only one that needs it.  Larger ones go through a pinned slot and a copy.
    PlanRef ref;
    HostPlan hp;
    PlanSlot* slot = nullptr;
    const size_t bytes = layout_of(pl, u.stage.size(), &ref);
    const bool fused = c->fused_combine && (size_t)pl.n_part_slots * desc->num_kv_heads * sizeof(uint32_t) <= kCounterBytes;
    alignas(16) uint8_t inline_plan[kMidPlanBytes];
    if (bytes <= (size_t)(pl.prefill_tc.empty() ? kMidPlanBytes : kSmallPlanBytes) && (fused || pl.combine.empty()) && !pl.pair) {
        write_plan(inline_plan, pl, u.stage, ref);
        hp.bytes = inline_plan;
        hp.size = bytes;
    } else {
        cf_status st = next_slot(c, bytes, &slot);
        if (st != CF_OK) return st;
        write_plan(slot->host, pl, u.stage, ref);
        st = upload_slot(slot, bytes, copy_stream, stream);
        if (st != CF_OK) return st;
        ref.base = slot->dev;
    }
    PlanCounts n;
    n.n_dec = (int)pl.decode.size(); n.n_comb = (int)pl.combine.size(); n.n_shared = (int)pl.shared_decode.size();
    n.n_pre_tc = (int)pl.prefill_tc.size(); n.n_pre_comb = (int)pl.prefill_combine.size(); n.total_q = pl.total_q;
    n.n_part_slots = pl.n_part_slots;
    n.pair = pl.pair;
    n.n_stage_seqs = (int)u.stage.size(); n.n_stage_pages = u.n_stage_pages; n.max_stage_pages = u.max_stage_pages; n.num_seqs = u.num_seqs;
    c->last_counts[0] = n.n_dec; c->last_counts[1] = n.n_comb; c->last_counts[2] = n.n_pre_tc; c->last_counts[3] = n.n_part_slots;
    c->last_counts[4] = n.n_pre_comb; c->last_counts[5] = shared_units(pl, desc); c->last_counts[6] = (int32_t)pl.share_members.size();
    c->last_counts[7] = pl.pair ? 1 : 0;
    n.front_sms = u.front_sms;
    const cf_status ls = launch_attention(c, desc, n, ref, hp, c->queue_dev, c->workspace, u.W, q, k_cache, v_cache, block_table,
                                          u.max_blocks, out, lse, stream, u.serial, true);
    const cf_status fs = slot ? finish_slot(slot, stream) : CF_OK;
    return ls != CF_OK ? ls : fs;
}

}  // namespace cf

extern "C" {

cf_status cf_kv_append(cf_ctx* c, const cf_cache_desc* desc, void* k_cache, void* v_cache,
                       const void* k_new, const void* v_new,
                       const int32_t* block_table, int32_t max_blocks_per_seq,
                       const int32_t* context_len, const int32_t* query_len,
                       int32_t num_seqs, void* cuda_stream)
{
    if (!c || !desc) return CF_ERR_INVALID_ARG;
    const int64_t t_in = now_ns();
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    Plan pl;
    st = validate_lengths(desc, context_len, query_len, num_seqs, max_blocks_per_seq, &pl);
    if (st != CF_OK) return st;
    if (pl.total_q == 0) return CF_OK;
    if (!k_cache || !v_cache || !k_new || !v_new || !block_table) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    st = enqueue_append(c, desc, pl, k_cache, v_cache, k_new, v_new, block_table, max_blocks_per_seq, context_len, query_len, num_seqs,
                        c->upload_stream, (cudaStream_t)cuda_stream);
    c->host_ns_append += now_ns() - t_in;
    ++c->host_calls_append;
    return st;
}

cf_status cf_mixed_attention(cf_ctx* c, const cf_cache_desc* desc, const void* q,
                             const void* k_cache, const void* v_cache,
                             const int32_t* block_table, int32_t max_blocks_per_seq,
                             const int32_t* context_len, const int32_t* query_len, int32_t num_seqs,
                             void* out, float* lse, void* cuda_stream)
{
    return cf_mixed_attention_shared(c, desc, q, k_cache, v_cache, block_table, max_blocks_per_seq, context_len, query_len,
                                     nullptr, nullptr, num_seqs, out, lse, cuda_stream);
}

cf_status cf_mixed_attention_shared(cf_ctx* c, const cf_cache_desc* desc, const void* q,
                                    const void* k_cache, const void* v_cache,
                                    const int32_t* block_table, int32_t max_blocks_per_seq,
                                    const int32_t* context_len, const int32_t* query_len,
                                    const int32_t* share_group, const int32_t* shared_len, int32_t num_seqs,
                                    void* out, float* lse, void* cuda_stream)
{
    if (!c || !desc) return CF_ERR_INVALID_ARG;
    if ((share_group == nullptr) != (shared_len == nullptr)) return CF_ERR_INVALID_ARG;
    const int64_t t_in = now_ns();
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    Unit u;
    st = validate_lengths(desc, context_len, query_len, num_seqs, max_blocks_per_seq, &u.pl);
    if (st != CF_OK) return st;
    c->launches = 0;
    if (u.pl.total_q == 0) return CF_OK;
    if (!q || !k_cache || !v_cache || !block_table || !out) return CF_ERR_INVALID_ARG;
    st = plan_unit(c, desc, context_len, query_len, num_seqs, max_blocks_per_seq, share_group, shared_len, false, &u);
    if (st != CF_OK) return st;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    st = ensure_workspace(c, u.W.total);
    if (st != CF_OK) return st;
    st = enqueue_unit(c, desc, u, q, k_cache, v_cache, block_table, out, lse, c->upload_stream, (cudaStream_t)cuda_stream);
    c->host_ns_attention += now_ns() - t_in;
    ++c->host_calls_attention;
    return st;
}

cf_status cf_plan_create(cf_ctx* c, const cf_cache_desc* desc, const int32_t* context_len, const int32_t* query_len,
                         int32_t num_seqs, int32_t max_blocks_per_seq, void* cuda_stream, cf_plan** out)
{
    if (!c || !desc || !out) return CF_ERR_INVALID_ARG;
    *out = nullptr;
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    Plan pl;
    PlanConfig cfg = c->cfg;
    const int front_sms = !c->overlap ? 0 : c->spatial_sms > 0 ? c->spatial_sms : spatial_front_sms(desc, context_len, query_len, num_seqs, c->num_sms);
    cfg.prefill_sms_mixed = front_sms;
    cfg.prefill_pair = c->use_pairs && prefill_pair_supported(desc);
    st = build_plan(desc, context_len, query_len, num_seqs, max_blocks_per_seq, cfg, &pl);
    if (st != CF_OK) return st;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    cf_plan* P = new (std::nothrow) cf_plan();
    if (!P) return CF_ERR_CUDA;
    P->ctx = c;
    P->desc = *desc;
    P->num_seqs = num_seqs;
    P->max_blocks = max_blocks_per_seq;
    std::vector<StageSeq> stage;
    int n_stage_pages = 0, max_stage_pages = 0;
    if (!pl.prefill_tc.empty()) stage_list(desc, context_len, query_len, num_seqs, &stage, &n_stage_pages, &max_stage_pages);
    P->off_len = align_up(layout_of(pl, stage.size(), &P->ref), 16);
    const size_t qs_bytes = sizeof(int32_t) * ((size_t)num_seqs + 1), pf_bytes = sizeof(int32_t) * (size_t)num_seqs;
    P->off_queue = align_up(P->off_len + qs_bytes + pf_bytes, 16);
    P->total = P->off_queue + 16;
    P->n_stage_seqs = (int)stage.size(); P->n_stage_pages = n_stage_pages; P->max_stage_pages = max_stage_pages;
    P->n_dec = (int)pl.decode.size(); P->n_comb = (int)pl.combine.size();
    P->n_pre_tc = (int)pl.prefill_tc.size(); P->n_pre_comb = (int)pl.prefill_combine.size(); P->total_q = pl.total_q;
    P->front_sms = c->spatial_sms > 0 ? front_sms : pl.front_sms;
    P->n_part_slots = pl.n_part_slots; P->n_pre_slots = pl.n_pre_slots;
    P->pair = pl.pair;
    const size_t part_bytes = ws_layout(pl.n_part_slots, pl.n_pre_slots, desc->num_q_heads, desc->head_dim, n_stage_pages,
                                        desc->num_kv_heads, (int64_t)num_seqs * max_blocks_per_seq).total;
    bool ok = cudaMallocHost((void**)&P->host, P->total) == cudaSuccess && cudaMalloc((void**)&P->dev, P->total) == cudaSuccess;
    // the ticket counters are zeroed on the caller's stream, like the plan copy: every launch that uses the plan
    // is ordered behind this call on that stream (or by the caller)
    if (ok && part_bytes)
        ok = cudaMalloc((void**)&P->part, part_bytes) == cudaSuccess &&
             cudaMemsetAsync(P->part, 0, kCounterBytes, (cudaStream_t)cuda_stream) == cudaSuccess;
    if (ok) {
        for (int32_t i = 0; i < num_seqs; ++i) pl.prefix.push_back(context_len[i] - query_len[i]);
        write_plan(P->host, pl, stage, P->ref);
        std::memcpy(P->host + P->off_len, pl.q_start.data(), qs_bytes);
        if (pf_bytes) std::memcpy(P->host + P->off_len + qs_bytes, pl.prefix.data(), pf_bytes);
        std::memset(P->host + P->off_queue, 0, 16);
        P->ref.base = P->dev;
        ok = cudaMemcpyAsync(P->dev, P->host, P->total, cudaMemcpyHostToDevice, (cudaStream_t)cuda_stream) == cudaSuccess;
    }
    c->live_plans.fetch_add(1);
    if (!ok) {
        cf_plan_destroy(P);
        return CF_ERR_CUDA;
    }
    *out = P;
    return CF_OK;
}

cf_status cf_plan_destroy(cf_plan* P)
{
    if (!P) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(P->ctx->device);
    cudaDeviceSynchronize();
    if (P->host) cudaFreeHost(P->host);
    if (P->dev) cudaFree(P->dev);
    if (P->part) cudaFree(P->part);
    P->ctx->live_plans.fetch_sub(1);
    delete P;
    return CF_OK;
}

cf_status cf_kv_append_planned(cf_plan* P, void* k_cache, void* v_cache, const void* k_new, const void* v_new,
                               const int32_t* block_table, void* cuda_stream)
{
    if (!P) return CF_ERR_INVALID_ARG;
    if (P->total_q == 0) return CF_OK;
    if (!k_cache || !v_cache || !k_new || !v_new || !block_table) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(P->ctx->device);
    if (!guard.ok) return CF_ERR_CUDA;
    AppendParams p = append_params(P->ctx, &P->desc, k_cache, v_cache, k_new, v_new, block_table, P->max_blocks, P->num_seqs, P->total_q);
    const size_t qs_bytes = sizeof(int32_t) * ((size_t)P->num_seqs + 1);
    if (P->num_seqs <= kAppendInlineSeqs) {
        p.host_q_start = (const int32_t*)(P->host + P->off_len);
        p.host_prefix = (const int32_t*)(P->host + P->off_len + qs_bytes);
    } else {
        p.q_start = (const int32_t*)(P->dev + P->off_len);
        p.prefix = (const int32_t*)(P->dev + P->off_len + qs_bytes);
    }
    return launch_kv_append(p, (cudaStream_t)cuda_stream) == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}

cf_status cf_mixed_attention_planned(cf_plan* P, const void* q, const void* k_cache, const void* v_cache,
                                     const int32_t* block_table, void* out, float* lse, void* cuda_stream)
{
    if (!P) return CF_ERR_INVALID_ARG;
    P->ctx->launches = 0;
    if (P->total_q == 0) return CF_OK;
    if (!q || !k_cache || !v_cache || !block_table || !out) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(P->ctx->device);
    if (!guard.ok) return CF_ERR_CUDA;
    PlanCounts n;
    n.n_dec = P->n_dec; n.n_comb = P->n_comb; n.n_pre_tc = P->n_pre_tc; n.n_pre_comb = P->n_pre_comb;
    n.total_q = P->total_q;
    n.front_sms = P->front_sms;
    n.n_part_slots = P->n_part_slots;
    n.pair = P->pair;
    n.n_stage_seqs = P->n_stage_seqs; n.n_stage_pages = P->n_stage_pages; n.max_stage_pages = P->max_stage_pages; n.num_seqs = P->num_seqs;
    const WsLayout W = ws_layout(P->n_part_slots, P->n_pre_slots, P->desc.num_q_heads, P->desc.head_dim, P->n_stage_pages,
                                 P->desc.num_kv_heads, (int64_t)P->num_seqs * P->max_blocks);
    return launch_attention(P->ctx, &P->desc, n, P->ref, HostPlan(), (uint32_t*)(P->dev + P->off_queue), P->part, W, q, k_cache,
                            v_cache, block_table, P->max_blocks, out, lse, (cudaStream_t)cuda_stream, false, false);
}

}  // extern "C"

namespace cf {

// A host-staged step in parts.  The result of a large chunk takes as long to cross the host link as a decode batch takes to
// compute (8 MB: 160 us at 52 GB/s), so a step whose prefill rows weigh enough is computed in parts, prefill first,
// and each part is read back while the next one runs; decode, which has next to nothing to read back, comes last.
// A part is a run of consecutive rows: whole sequences, or a chunk cut at a multiple of 128 rows (the rest of the
// chunk sees the same cache: the whole step has been appended before).  Measured per step, in one piece -> in parts: chat mix
// 484 -> 331 us, agentic mix 1164 -> 975 us, 512 rows beside 256 decodes on an fp8 cache 561 -> 424 us, 8192 rows beside 256
// decodes 4.20 -> 3.94 ms.
struct HostPart {
    int32_t seq = 0, num_seqs = 0;               // sequences [seq, seq + num_seqs)
    int64_t row = 0, rows = 0;                   // packed rows
    std::vector<int32_t> context_len, query_len;
    double us = 0.0;                             // estimated time on the device
};

// Parts of the step, or none when it is better computed and read back as one: few bytes, or too many runs.
// *kernel_bound: the kernels outweigh both directions of the link.
static std::vector<HostPart> host_parts(const cf_cache_desc* d, const int32_t* context_len, const int32_t* query_len, int32_t S,
                                        const std::vector<int32_t>& q_start, int num_sms, bool* kernel_bound)
{
    constexpr double kMinPrefillBytes = 4 << 20;      // below: the read-back is shorter than what the parts cost
    constexpr double kLinkBytesPerUs = 52e3, kPartUs = 12.0;
    constexpr int32_t kMaxRuns = 4, kMaxCuts = 4;
    const int32_t G = d->num_q_heads / d->num_kv_heads, W = d->window_size;
    const double row_bytes = 2.0 * d->num_q_heads * d->head_dim;
    std::vector<HostPart> runs[2];                    // prefill, decode: runs of consecutive sequences of one kind
    int last = -1;
    for (int32_t s = 0; s < S; ++s) {
        const int32_t lq = query_len[s], lc = context_len[s];
        const int kind = lq == 0 ? last : lq == 1 ? 1 : 0;
        if (kind < 0) continue;
        if (kind != last) {
            runs[kind].emplace_back();
            runs[kind].back().seq = s;
            runs[kind].back().row = q_start[(size_t)s];
            last = kind;
        }
        HostPart& r = runs[kind].back();
        r.num_seqs = s + 1 - r.seq;
        r.rows += lq;
        r.context_len.push_back(lc);
        r.query_len.push_back(lq);
        // rough device time: decode streams its cache, prefill is items of 256 / G rows at the machine's average
        if (lq == 1) r.us += 2.0 * (W > 0 ? std::min(lc, W) : lc) * d->num_kv_heads * d->head_dim * (d->kv_dtype == CF_KV_FP8_E4M3 ? 1 : 2) / 6.5e6;
        else if (lq > 1)
            for (int32_t at = 0; at < lq; at += 128) {
                const int32_t hi = lc - lq + std::min(lq, at + 128), lo = W > 0 ? std::max(0, lc - lq + at - W + 1) : 0;
                r.us += (double)d->num_kv_heads * ((std::min(128, lq - at) * G + 255) / 256) * (5.0 + 1.8 * ((hi - lo + 127) / 128)) / num_sms;
            }
    }
    double pre_rows = 0.0, pre_us = 0.0, dec_us = 0.0;
    for (const HostPart& r : runs[0]) { pre_rows += (double)r.rows; pre_us += r.us; }
    for (const HostPart& r : runs[1]) dec_us += r.us;
    std::vector<HostPart> parts;
    if (pre_rows * row_bytes < kMinPrefillBytes || runs[0].size() + runs[1].size() > (size_t)kMaxRuns) return parts;
    // A step whose inputs take longer to cross the link than all of this is bound by them (three ragged chunks of 5003 rows:
    // 61 MB in, 41 MB out, 1350 us either way; in parts the two directions get in each other's way, +3 %).
    const double link_us = pre_rows * row_bytes / kLinkBytesPerUs;
    const double in_us = ((double)q_start.back() * (row_bytes + 4.0 * d->num_kv_heads * d->head_dim)) / kLinkBytesPerUs;
    if (in_us > pre_us + dec_us + link_us) return parts;
    *kernel_bound = pre_us + dec_us > 1.25 * std::max(in_us, link_us);
    // how many pieces to cut the prefill rows into: the end of the last read-back, all pieces taken as equal
    int32_t cuts = 1;
    double best = 1e30;
    for (int32_t n = 1; n <= kMaxCuts; ++n) {
        const double piece = pre_us / n + kPartUs;
        double link = 0.0;
        for (int32_t i = 1; i <= n; ++i) link = std::max(link, i * piece) + link_us / n;
        const double end = std::max(link, n * piece + dec_us);
        if (end < best * 0.97) { best = end; cuts = n; }
    }
    const int64_t piece_rows = ((int64_t)(pre_rows / cuts) + 127) / 128 * 128;
    for (const HostPart& r : runs[0]) {
        HostPart cur;
        auto close = [&] {
            if (cur.rows > 0) parts.push_back(std::move(cur));
            cur = HostPart();
        };
        int64_t row = r.row;
        for (int32_t i = 0; i < r.num_seqs; ++i) {
            const int32_t lq = r.query_len[(size_t)i], prefix = r.context_len[(size_t)i] - lq;
            for (int32_t a = 0; a < lq;) {
                // up to the piece's size, on a 128-row boundary of the chunk; a short rest stays with the piece
                int64_t take = std::max<int64_t>(128, (piece_rows - cur.rows) / 128 * 128);
                if (lq - a - take < 128) take = lq - a;
                if (cur.rows == 0) { cur.seq = r.seq + i; cur.row = row; }
                cur.num_seqs = r.seq + i + 1 - cur.seq;
                while ((int32_t)cur.query_len.size() < cur.num_seqs - 1) {     // sequences without new rows in between
                    cur.context_len.push_back(0);
                    cur.query_len.push_back(0);
                }
                cur.context_len.push_back(prefix + a + (int32_t)take);
                cur.query_len.push_back((int32_t)take);
                cur.rows += take;
                row += take;
                a += (int32_t)take;
                if (cur.rows >= piece_rows || a < lq) close();        // a sequence has one entry per part
            }
        }
        close();
    }
    for (HostPart& r : runs[1]) parts.push_back(std::move(r));
    if (parts.size() > (size_t)kHostParts) parts.clear();
    return parts;
}

// The planned parts of a step as one call (join_plans); false where it does not fit a fixed workspace.
static bool join_units(cf_ctx* c, const cf_cache_desc* desc, const std::vector<HostPart>& parts, const std::vector<Unit>& units,
                       const int32_t* context_len, const int32_t* query_len, int32_t num_seqs, int32_t max_blocks_per_seq, Unit* u)
{
    std::vector<const Plan*> plans;
    std::vector<int32_t> seqs;
    std::vector<int64_t> rows;
    for (size_t i = 0; i < parts.size(); ++i) {
        plans.push_back(&units[i].pl);
        seqs.push_back(parts[i].seq);
        rows.push_back(parts[i].row);
    }
    join_plans(desc, plans, seqs, rows, &u->pl);
    stage_list(desc, context_len, query_len, num_seqs, &u->stage, &u->n_stage_pages, &u->max_stage_pages);
    u->W = ws_layout(u->pl.n_part_slots, u->pl.n_pre_slots, desc->num_q_heads, desc->head_dim, u->n_stage_pages, desc->num_kv_heads,
                     (int64_t)num_seqs * max_blocks_per_seq);
    u->num_seqs = num_seqs;
    u->max_blocks = max_blocks_per_seq;
    u->front_sms = spatial_front_sms(desc, context_len, query_len, num_seqs, c->num_sms);
    u->serial = u->front_sms <= (c->num_sms * 3) / 5;      // as for a step that is not cut
    return !c->workspace_fixed || u->W.total <= c->workspace_bytes;
}

}  // namespace cf

extern "C" {

cf_status cf_mixed_step_host(cf_ctx* c, const cf_cache_desc* desc,
                             const void* q_host, const void* k_new_host, const void* v_new_host,
                             void* k_cache, void* v_cache,
                             const int32_t* block_table, int32_t max_blocks_per_seq,
                             const int32_t* context_len, const int32_t* query_len, int32_t num_seqs,
                             void* out_host, void* cuda_stream)
{
    if (!c || !desc) return CF_ERR_INVALID_ARG;
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    Plan pl;
    st = validate_lengths(desc, context_len, query_len, num_seqs, max_blocks_per_seq, &pl);
    if (st != CF_OK) return st;
    if (pl.total_q == 0) return CF_OK;
    if (!q_host || !k_new_host || !v_new_host || !out_host || !k_cache || !v_cache || !block_table) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    cudaStream_t stream = (cudaStream_t)cuda_stream;

    // Plans the step, all of its parts.  With a fixed workspace this comes before anything is enqueued: a part that does not fit
    // refuses the step while the caches and out_host are as they were.  A growing workspace refuses nothing, and the planning
    // runs beside the input copies (a step that is waited for: chat mix 581 -> 566 us, 512 rows on an fp8 cache 723 -> 697 us).
    const int64_t t_in = now_ns();
    std::vector<HostPart> parts;
    std::vector<Unit> units;
    bool whole = false;
    auto plan = [&]() -> cf_status {
        bool kernel_bound = false;
        parts = host_parts(desc, context_len, query_len, num_seqs, pl.q_start, c->num_sms, &kernel_bound);
        whole = parts.empty();
        units.resize(whole ? 1 : parts.size());
        size_t ws_bytes = 0;
        for (size_t i = 0; i < units.size(); ++i) {
            // In one piece: a step whose decode part weighs as much as its prefill part is bound by the copies over the host link,
            // not by the kernels, and keeps the serial sequence; a prefill-heavy step (the spatial share above its floor) runs
            // the sequence cf_mixed_attention would run.
            const cf_status e = whole ? plan_unit(c, desc, context_len, query_len, num_seqs, max_blocks_per_seq, nullptr, nullptr,
                                                  spatial_front_sms(desc, context_len, query_len, num_seqs, c->num_sms) <= (c->num_sms * 3) / 5, &units[i])
                                      : plan_unit(c, desc, parts[i].context_len.data(), parts[i].query_len.data(), parts[i].num_seqs,
                                                  max_blocks_per_seq, nullptr, nullptr, true, &units[i]);
            if (e != CF_OK) return e;
            ws_bytes = std::max(ws_bytes, units[i].W.total);
        }
        // A step that follows another without a flush in between has its read-back under the kernels of the next one anyway.
        // Where the kernels outweigh both directions of the link such steps are bound by them, and the parts' items run as one
        // call, decode beside prefill (agentic, back to back, in parts 1006 us per step, as one call 914); where the link weighs as
        // much, parts still help.  The items are the parts' own (decode in chunks for all SMs, as it runs alone in parts), so a step's
        // result does not depend on the steps before it.
        if (!whole && kernel_bound && c->unflushed_steps > 0) {
            Unit u;
            if (join_units(c, desc, parts, units, context_len, query_len, num_seqs, max_blocks_per_seq, &u)) {
                units.clear();
                units.push_back(std::move(u));
                ws_bytes = units[0].W.total;
                whole = true;
            }
        }
        return ensure_workspace(c, ws_bytes);
    };
    if (c->workspace_fixed && (st = plan()) != CF_OK) return st;
    c->launches = 0;

    const size_t T = (size_t)pl.total_q;
    const size_t q_bytes = align_up(T * desc->num_q_heads * desc->head_dim * 2, 256);
    const size_t kv_bytes = align_up(T * desc->num_kv_heads * desc->head_dim * 2, 256);
    const size_t need = 2 * q_bytes + 2 * kv_bytes;
    HostStage& hs = c->stage[c->next_stage];
    if (need > hs.bytes) {
        if (cudaDeviceSynchronize() != cudaSuccess) return CF_ERR_CUDA;
        if (hs.dev) cudaFree(hs.dev);
        hs.dev = nullptr;
        hs.bytes = 0;
        if (cudaMalloc((void**)&hs.dev, need) != cudaSuccess) return CF_ERR_CUDA;
        hs.bytes = need;
        hs.used = false;
    }
    c->next_stage = (c->next_stage + 1) % kHostStages;
    uint8_t* dq = hs.dev;
    uint8_t* dk = dq + q_bytes;
    uint8_t* dv = dk + kv_bytes;
    uint8_t* dout = dv + kv_bytes;
    const size_t row_bytes = (size_t)desc->num_q_heads * desc->head_dim * 2;
    const size_t qb = T * row_bytes, kb = T * desc->num_kv_heads * desc->head_dim * 2;
    auto run = [&]() -> cf_status {
        auto ok = [](cudaError_t e) { return e == cudaSuccess; };
        // inputs: copy stream, after the kernels and the read-back that last used this staging set
        // (q on one copy stream, k_new and v_new on a second: the small copies run at two thirds of the link rate
        // on their own and fill in beside the large one)
        if (hs.used && !(ok(cudaStreamWaitEvent(c->h2d_stream, hs.compute_done, 0)) && ok(cudaStreamWaitEvent(c->h2d_stream, hs.d2h_done, 0)) &&
                         ok(cudaStreamWaitEvent(c->h2d_kv_stream, hs.compute_done, 0))))
            return CF_ERR_CUDA;
        if (!ok(cudaMemcpyAsync(dk, k_new_host, kb, cudaMemcpyHostToDevice, c->h2d_kv_stream)) ||
            !ok(cudaMemcpyAsync(dv, v_new_host, kb, cudaMemcpyHostToDevice, c->h2d_kv_stream)) ||
            !ok(cudaEventRecord(hs.h2d_kv_done, c->h2d_kv_stream)) ||
            !ok(cudaMemcpyAsync(dq, q_host, qb, cudaMemcpyHostToDevice, c->h2d_stream)) || !ok(cudaEventRecord(hs.h2d_done, c->h2d_stream)))
            return CF_ERR_CUDA;
        cf_status e = c->workspace_fixed ? CF_OK : plan();
        if (e != CF_OK) return e;
        // kernels: the caller's stream; plans are uploaded on the input copy stream
        if (!ok(cudaStreamWaitEvent(stream, hs.h2d_kv_done, 0))) return CF_ERR_CUDA;
        e = enqueue_append(c, desc, pl, k_cache, v_cache, dk, dv, block_table, max_blocks_per_seq, context_len, query_len, num_seqs,
                                     c->h2d_stream, stream);
        if (e != CF_OK) return e;
        if (!ok(cudaStreamWaitEvent(stream, hs.h2d_done, 0))) return CF_ERR_CUDA;
        for (size_t i = 0; i < units.size(); ++i) {
            const size_t off = whole ? 0 : (size_t)parts[i].row * row_bytes, bytes = whole ? qb : (size_t)parts[i].rows * row_bytes;
            const int32_t* table = whole ? block_table : block_table + (int64_t)parts[i].seq * max_blocks_per_seq;
            e = enqueue_unit(c, desc, units[i], dq + off, k_cache, v_cache, table, dout + off, nullptr, c->h2d_stream, stream);
            if (e != CF_OK) return e;
            // result: second copy stream
            if (!ok(cudaEventRecord(hs.part_done[i], stream)) || !ok(cudaStreamWaitEvent(c->d2h_stream, hs.part_done[i], 0)) ||
                !ok(cudaMemcpyAsync((uint8_t*)out_host + off, dout + off, bytes, cudaMemcpyDeviceToHost, c->d2h_stream)))
                return CF_ERR_CUDA;
        }
        return CF_OK;
    };
    st = run();
    // Also where a call failed half-way: what has been enqueued is ordered before the staging set's next use and before the flush.
    if (st != CF_OK) {
        cudaEventRecord(hs.h2d_done, c->h2d_stream);
        cudaEventRecord(hs.h2d_kv_done, c->h2d_kv_stream);
        cudaStreamWaitEvent(stream, hs.h2d_done, 0);
        cudaStreamWaitEvent(stream, hs.h2d_kv_done, 0);
    }
    const bool done = cudaEventRecord(hs.compute_done, stream) == cudaSuccess &&
                      (st == CF_OK || cudaStreamWaitEvent(c->d2h_stream, hs.compute_done, 0) == cudaSuccess) &&
                      cudaEventRecord(hs.d2h_done, c->d2h_stream) == cudaSuccess;
    hs.used = true;
    c->host_ns_attention += now_ns() - t_in;
    c->host_calls_append += 1;
    c->host_calls_attention += (int32_t)units.size();
    if (st == CF_OK && !done) st = CF_ERR_CUDA;
    if (st == CF_OK) ++c->unflushed_steps;
    return st;
}

cf_status cf_host_steps_flush(cf_ctx* c, void* cuda_stream)
{
    if (!c) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    for (int i = 0; i < kHostStages; ++i)
        if (c->stage[i].used && cudaStreamWaitEvent((cudaStream_t)cuda_stream, c->stage[i].d2h_done, 0) != cudaSuccess)
            return CF_ERR_CUDA;
    c->unflushed_steps = 0;
    return CF_OK;
}

cf_status cf_get_async_status(cf_ctx* c)
{
    if (!c) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    uint32_t w = 0;
    if (cudaMemcpy(&w, c->err_dev, sizeof w, cudaMemcpyDeviceToHost) != cudaSuccess) return CF_ERR_CUDA;
    if (w == 0) return CF_OK;
    if (cudaMemset(c->err_dev, 0, sizeof w) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return CF_ERR_CUDA;
    if (w & kErrTimeout) return CF_ERR_TIMEOUT;
    if (w & kErrBlockId) return CF_ERR_OUT_OF_RANGE;
    return CF_ERR_CUDA;
}

cf_status cf_validate_block_table(cf_ctx* c, const cf_cache_desc* desc, const int32_t* block_table,
                                  int32_t max_blocks_per_seq, const int32_t* context_len, const int32_t* query_len,
                                  int32_t num_seqs, void* cuda_stream, int32_t* num_bad)
{
    if (!c || !desc || !num_bad) return CF_ERR_INVALID_ARG;
    *num_bad = 0;
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    Plan pl;
    st = validate_lengths(desc, context_len, query_len, num_seqs, max_blocks_per_seq, &pl);
    if (st != CF_OK) return st;
    if (num_seqs == 0) return CF_OK;
    if (!block_table) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    PlanSlot* slot = nullptr;
    const size_t bytes = sizeof(int32_t) * (size_t)num_seqs;
    st = next_slot(c, bytes, &slot);
    if (st != CF_OK) return st;
    std::memcpy(slot->host, context_len, bytes);
    st = upload_slot(slot, bytes, c->upload_stream, stream);
    if (st != CF_OK) return st;
    uint32_t* counter = c->err_dev + 1;      // context-owned scratch word
    bool ok = cudaMemsetAsync(counter, 0, sizeof(uint32_t), stream) == cudaSuccess;
    ok = ok && launch_validate_table(block_table, max_blocks_per_seq, (const int32_t*)slot->dev, num_seqs,
                                     desc->num_blocks, counter, stream) == cudaSuccess;
    finish_slot(slot, stream);
    uint32_t host = 0;
    ok = ok && cudaMemcpyAsync(&host, counter, sizeof host, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(stream) == cudaSuccess;
    if (!ok) return CF_ERR_CUDA;
    *num_bad = (int32_t)host;
    return host ? CF_ERR_OUT_OF_RANGE : CF_OK;
}

cf_status cf_set_overlap(cf_ctx* c, int enabled)
{
    if (!c) return CF_ERR_INVALID_ARG;
    if (enabled < 0) return CF_ERR_INVALID_ARG;
    c->overlap = enabled != 0;
    if (enabled > 1) c->spatial_sms = enabled;
    if (enabled == 1) c->spatial_sms = c->spatial_sms_default;
    return CF_OK;
}

cf_status cf_set_debug_option(cf_ctx* c, cf_debug_option option, int value)
{
    if (!c) return CF_ERR_INVALID_ARG;
    const PlanConfig defaults;
    switch (option) {
        case CF_DEBUG_PREFILL_SPLIT: c->cfg.prefill_force_split = value > 0 ? value : 0; return CF_OK;
        case CF_DEBUG_SEPARATE_COMBINE: c->fused_combine = value <= 0; return CF_OK;
        case CF_DEBUG_DECODE_WAVES: c->cfg.decode_waves = value > 0 ? value : defaults.decode_waves; return CF_OK;
        case CF_DEBUG_DECODE_MIN_CHUNK_PAGES:
            c->cfg.decode_min_chunk_pages = value > 0 ? value : defaults.decode_min_chunk_pages;
            return CF_OK;
        case CF_DEBUG_SPATIAL_NO_WAIT: return CF_OK;      // no effect: the launches themselves carry the order
        case CF_DEBUG_PREFILL_PAIRS: c->use_pairs = value > 0; return CF_OK;
    }
    return CF_ERR_INVALID_ARG;
}

cf_status cf_selftest_bounded_wait(cf_ctx* c, void* cuda_stream)
{
    if (!c) return CF_ERR_INVALID_ARG;
    DeviceGuard guard(c->device);
    if (!guard.ok) return CF_ERR_CUDA;
    return launch_wait_selftest(c->err_dev, (cudaStream_t)cuda_stream) == cudaSuccess ? CF_OK : CF_ERR_CUDA;
}

cf_status cf_set_timing(cf_ctx* c, int enabled)
{
    if (!c) return CF_ERR_INVALID_ARG;
    c->timing = enabled != 0;
    c->timed_used = 0;
    return CF_OK;
}

cf_status cf_get_timing_sums(cf_ctx* c, float* ms_decode, float* ms_combine, float* ms_prefill, int32_t* num_calls)
{
    if (!c) return CF_ERR_INVALID_ARG;
    double t[3] = {0., 0., 0.};
    const size_t n = c->timed_used;
    if (n > 0) {
        DeviceGuard guard(c->device);
        if (cudaEventSynchronize(c->timed[n - 1].ev[3]) != cudaSuccess) return CF_ERR_CUDA;
        for (size_t k = 0; k < n; ++k)
            for (int i = 0; i < 3; ++i) {
                float ms = 0.f;
                if (c->timed[k].ran[i] && cudaEventElapsedTime(&ms, c->timed[k].ev[i], c->timed[k].ev[i + 1]) != cudaSuccess)
                    return CF_ERR_CUDA;
                t[i] += ms;
            }
    }
    c->timed_used = 0;
    if (ms_decode) *ms_decode = (float)t[0];
    if (ms_combine) *ms_combine = (float)t[1];
    if (ms_prefill) *ms_prefill = (float)t[2];
    if (num_calls) *num_calls = (int32_t)n;
    return CF_OK;
}

cf_status cf_get_host_time_sums(cf_ctx* c, double* us_append, double* us_attention, double* us_planner, int32_t* num_steps)
{
    if (!c) return CF_ERR_INVALID_ARG;
    if (us_append) *us_append = 1e-3 * (double)c->host_ns_append;
    if (us_attention) *us_attention = 1e-3 * (double)c->host_ns_attention;
    if (us_planner) *us_planner = 1e-3 * (double)c->host_ns_planner;
    if (num_steps) *num_steps = c->host_calls_attention;
    c->host_ns_append = c->host_ns_attention = c->host_ns_planner = 0;
    c->host_calls_append = c->host_calls_attention = 0;
    return CF_OK;
}

cf_status cf_get_last_plan_counts(cf_ctx* c, int32_t* counts)
{
    if (!c || !counts) return CF_ERR_INVALID_ARG;
    for (int i = 0; i < 8; ++i) counts[i] = c->last_counts[i];
    return CF_OK;
}

cf_status cf_get_last_launch_count(cf_ctx* c, int32_t* num_launches)
{
    if (!c || !num_launches) return CF_ERR_INVALID_ARG;
    *num_launches = c->launches;
    return CF_OK;
}

int32_t cf_spatial_share(const cf_cache_desc* desc, const int32_t* context_len, const int32_t* query_len,
                         int32_t num_seqs, int32_t num_sms)
{
    if (validate_desc(desc) != CF_OK || num_seqs < 0 || (num_seqs > 0 && (!context_len || !query_len))) return 0;
    return spatial_front_sms(desc, context_len, query_len, num_seqs, num_sms > 0 ? num_sms : 148);
}

cf_status cf_estimate_us(const cf_cache_desc* desc, const int32_t* context_len, const int32_t* query_len,
                         int32_t num_seqs, int32_t max_blocks_per_seq, int32_t num_sms,
                         float* us_decode, float* us_combine, float* us_prefill)
{
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    PlanConfig cfg;
    cfg.num_sms = num_sms > 0 ? num_sms : 148;
    Plan pl;
    st = build_plan(desc, context_len, query_len, num_seqs, max_blocks_per_seq, cfg, &pl);
    if (st != CF_OK) return st;
    const Estimate e = estimate_us(desc, context_len, query_len, pl, cfg.num_sms);
    if (us_decode) *us_decode = e.us_decode;
    if (us_combine) *us_combine = e.us_combine;
    if (us_prefill) *us_prefill = e.us_prefill;
    return CF_OK;
}

cf_status cf_plan_inspect(const cf_cache_desc* desc, const int32_t* context_len, const int32_t* query_len,
                          int32_t num_seqs, int32_t max_blocks_per_seq, const cf_plan_options* opts,
                          int32_t* decode_items, int32_t* combine_items, int32_t* prefill_items,
                          int32_t cap, int32_t* counts)
{
    cf_status st = validate_desc(desc);
    if (st != CF_OK) return st;
    PlanConfig cfg;
    if (opts) {
        if (opts->num_sms > 0) cfg.num_sms = opts->num_sms;
        if (opts->prefill_sms_mixed > 0) cfg.prefill_sms_mixed = opts->prefill_sms_mixed;
        if (opts->prefill_force_split > 0) cfg.prefill_force_split = opts->prefill_force_split;
        if (opts->decode_waves > 0) cfg.decode_waves = opts->decode_waves;
        if (opts->decode_min_chunk_pages > 0) cfg.decode_min_chunk_pages = opts->decode_min_chunk_pages;
    }
    cfg.prefill_pair = prefill_pair_supported(desc) && opts && opts->prefill_pairs > 0;
    Plan pl;
    st = build_plan(desc, context_len, query_len, num_seqs, max_blocks_per_seq, cfg, &pl);
    if (st != CF_OK) return st;
    if (cap < 0) cap = 0;
    if (decode_items)
        for (size_t i = 0; i < pl.decode.size() && i < (size_t)cap; ++i) {
            const DecodeItem& d = pl.decode[i];
            int32_t* o = decode_items + 6 * i;
            o[0] = d.seq; o[1] = d.q_row; o[2] = d.kv_begin; o[3] = d.kv_end; o[4] = d.part_slot; o[5] = d.chunk;
        }
    if (combine_items)
        for (size_t i = 0; i < pl.combine.size() && i < (size_t)cap; ++i) {
            int32_t* o = combine_items + 3 * i;
            o[0] = pl.combine[i].q_row; o[1] = pl.combine[i].part_first; o[2] = pl.combine[i].n_chunks;
        }
    static_assert(sizeof(PrefillEntry) == 8 * sizeof(int32_t), "copied out as rows of eight");
    const std::vector<PrefillEntry> entries = list_prefill(desc, pl);
    const size_t n_pre = entries.size();
    if (prefill_items && n_pre) std::memcpy(prefill_items, entries.data(), sizeof(PrefillEntry) * std::min(n_pre, (size_t)cap));
    if (counts) {
        counts[0] = (int32_t)pl.decode.size();
        counts[1] = (int32_t)pl.combine.size();
        counts[2] = (int32_t)n_pre;
        counts[3] = pl.n_part_slots;
        counts[4] = (int32_t)pl.prefill_tc.size();          // prefill CTAs, KV ranges of split items included
        counts[5] = (int32_t)pl.prefill_combine.size();     // KV-split prefill items
    }
    return CF_OK;
}

}  // extern "C"
