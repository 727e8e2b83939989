// KV append: scatters this iteration's new K/V rows into the paged cache through the block table.
// Pure 16-byte moves, bit-exact (an fp8 cache: 16 values are quantised per 16-byte store).
//
// Bound by HBM for a large chunk and by latency for a decode batch.  One warp moves one row of K and of V: its loads
// (up to eight 16-byte loads per lane in flight) depend on the row number alone and are issued first; the search for
// the row's sequence and the block-table entry run behind them.  The search takes one load per factor of 32 (all
// lanes look at one boundary each and vote) instead of one per factor of 2.  Back to back on a B200, against
// one CTA of 256 threads per row with the search first: 8448 rows of 8 x 128 among 260 sequences 22.5 -> 8.8 us (7.9 TB/s
// read + written, from L2), 5003 rows 10.3 -> 5.7 us, 4160 rows of 8 x 64 8.2 -> 4.5 us, 768 rows onto an fp8 cache
// 6.2 -> 5.0 us, 64 rows 5.1 -> 4.5 us (launch latency).
#include <cuda_fp16.h>

#include <cstring>

#include "kernels.h"

namespace cf {

namespace {

constexpr int kAppendWarps = 4;        // rows per CTA
constexpr int kAppendLoads = 8;        // 16-byte loads per lane in flight

// sequence owning packed row `row`: the last s in [0, n) with q_start[s] <= row (q_start is non-decreasing), by the
// whole warp
__device__ __forceinline__ int sequence_of_row(const int32_t* q_start, int n, int row, int lane)
{
    int lo = 0;
    while (n > 1) {
        const int step = (n + 31) >> 5, i = lane * step;
        const uint32_t below = __ballot_sync(0xffffffffu, i < n && q_start[lo + i] <= row);
        const int last = 31 - __clz(below);            // lane 0 always votes: q_start[lo] <= row
        lo += last * step;
        n = min(step, n - last * step);
    }
    return lo;
}

// Sixteen bf16 values (two 16-byte loads) -> sixteen e4m3 codes of x / scale.  The quotient is an IEEE fp32 division and
// the conversion rounds to nearest even and saturates: the code is an integer decision that the CPU definition takes
// in the same precision.
__device__ __forceinline__ uint4 quantise16(const uint4 a, const uint4 b, const float scale)
{
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t packed[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t out = 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t pair = w[2 * i + h];
            const float lo = __fdiv_rn(__uint_as_float(pair << 16), scale), hi = __fdiv_rn(__uint_as_float(pair & 0xffff0000u), scale);
            uint16_t two;
            asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(two) : "f"(hi), "f"(lo));     // first source -> upper byte
            out |= (uint32_t)two << (16 * h);
        }
        packed[i] = out;
    }
    return make_uint4(packed[0], packed[1], packed[2], packed[3]);
}

}  // namespace

// A unit is 16 bytes of the cache: 8 bf16 elements, or 16 codes made from two 16-byte loads.  Units of K, then of V.
// SEQS > 0: the lengths of a batch of up to SEQS sequences come with the launch (about 0.3 us per launch at 4 KB, measured)
// instead of through a copy that the kernel would have to wait for.
template <int SEQS>
struct AppendLengths {
    int32_t q_start[SEQS + 1], prefix[SEQS];
};
template <>
struct AppendLengths<0> {
    static constexpr const int32_t *q_start = nullptr, *prefix = nullptr;
};

template <int D, bool FP8, int SEQS>
__global__ void __launch_bounds__(kAppendWarps * 32) kv_append_kernel(const AppendParams p, const __grid_constant__ AppendLengths<SEQS> len)
{
    constexpr int PER_HEAD = D / (FP8 ? 16 : 8);       // units of one head's row
    constexpr int WORDS = FP8 ? 2 : 1;                 // 16-byte loads per unit
    constexpr int UNROLL = kAppendLoads / WORDS;
    constexpr int ELEM = FP8 ? 1 : 2;
    const int lane = threadIdx.x & 31, row = blockIdx.x * kAppendWarps + (threadIdx.x >> 5);
    // programmatic launch: set up beside the tail of the grid before, which may still read the cache or write the new rows
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (row >= p.total_rows) return;
    const int per_tensor = p.Hkv * PER_HEAD, units = 2 * per_tensor;
    const uint4* const src_k = reinterpret_cast<const uint4*>(p.k_new) + (int64_t)row * per_tensor * WORDS;
    const uint4* const src_v = reinterpret_cast<const uint4*>(p.v_new) + (int64_t)row * per_tensor * WORDS;
    int64_t blk = 0;
    int slot = 0;
    for (int u0 = 0; u0 < units; u0 += 32 * UNROLL) {
        uint4 in[UNROLL * WORDS];
#pragma unroll
        for (int i = 0; i < UNROLL; ++i) {
            const int u = u0 + i * 32 + lane;
            if (u < units) {
                const uint4* src = u < per_tensor ? src_k + u * WORDS : src_v + (u - per_tensor) * WORDS;
#pragma unroll
                for (int w = 0; w < WORDS; ++w) in[i * WORDS + w] = __ldg(src + w);
            }
        }
        if (u0 == 0) {
            const int32_t* const q_start = SEQS > 0 ? len.q_start : p.q_start;
            const int s = sequence_of_row(q_start, p.num_seqs, row, lane);
            const int pos = (SEQS > 0 ? len.prefix : p.prefix)[s] + row - q_start[s];
            blk = __ldg(p.block_table + (int64_t)s * p.max_blocks + (pos >> 4));
            slot = pos & 15;
            if (blk < 0 || blk >= p.num_blocks) {      // never write outside the pool
                if (lane == 0 && p.err) atomicOr(p.err, kErrBlockId);
                return;
            }
        }
        uint8_t* const dst_k = reinterpret_cast<uint8_t*>(p.k_cache) + (blk * p.ks_block + slot * p.ks_token) * ELEM;
        uint8_t* const dst_v = reinterpret_cast<uint8_t*>(p.v_cache) + (blk * p.vs_block + slot * p.vs_token) * ELEM;
#pragma unroll
        for (int i = 0; i < UNROLL; ++i) {
            const int u = u0 + i * 32 + lane;
            if (u < units) {
                const bool is_v = u >= per_tensor;
                const int t = is_v ? u - per_tensor : u, g = t / PER_HEAD, c = t % PER_HEAD;
                uint8_t* dst = is_v ? dst_v + g * p.vs_head * ELEM : dst_k + g * p.ks_head * ELEM;
                uint4 out = in[i * WORDS];
                if constexpr (FP8) out = quantise16(in[2 * i], in[2 * i + 1], __ldg((is_v ? p.v_scale : p.k_scale) + g));
                *reinterpret_cast<uint4*>(dst + c * 16) = out;
            }
        }
    }
}

// Debug aid: counts the block-table entries that a call with these lengths would dereference and that
// fall outside [0, num_blocks).  Reads the table only; never touches the caches.
__global__ void validate_table_kernel(const int32_t* block_table, int32_t max_blocks, const int32_t* context_len,
                                      int32_t num_seqs, int32_t num_blocks, uint32_t* bad_count)
{
    const int s = blockIdx.x;
    if (s >= num_seqs) return;
    const int used = (context_len[s] + 15) >> 4;
    uint32_t bad = 0;
    for (int i = threadIdx.x; i < used && i < max_blocks; i += blockDim.x) {
        const int32_t b = block_table[(int64_t)s * max_blocks + i];
        bad += (b < 0 || b >= num_blocks) ? 1u : 0u;
    }
    if (bad) atomicAdd(bad_count, bad);
}

cudaError_t launch_validate_table(const int32_t* block_table, int32_t max_blocks, const int32_t* context_len_dev,
                                  int32_t num_seqs, int32_t num_blocks, uint32_t* bad_count, cudaStream_t stream)
{
    if (num_seqs <= 0) return cudaSuccess;
    validate_table_kernel<<<num_seqs, 128, 0, stream>>>(block_table, max_blocks, context_len_dev, num_seqs, num_blocks, bad_count);
    return cudaGetLastError();
}

namespace {

template <int D, bool FP8, int SEQS>
cudaError_t launch_append_t(const AppendParams& p, const cudaLaunchConfig_t& cfg)
{
    AppendLengths<SEQS> len;
    if constexpr (SEQS > 0) {
        std::memcpy(len.q_start, p.host_q_start, sizeof(int32_t) * ((size_t)p.num_seqs + 1));
        std::memcpy(len.prefix, p.host_prefix, sizeof(int32_t) * (size_t)p.num_seqs);
    }
    return cudaLaunchKernelEx(&cfg, kv_append_kernel<D, FP8, SEQS>, p, len);
}
template <int D, bool FP8>
cudaError_t launch_append_d(const AppendParams& p, const cudaLaunchConfig_t& cfg)
{
    if (p.q_start != nullptr) return launch_append_t<D, FP8, 0>(p, cfg);
    return p.num_seqs <= 64 ? launch_append_t<D, FP8, 64>(p, cfg) : launch_append_t<D, FP8, kAppendInlineSeqs>(p, cfg);
}

}  // namespace

cudaError_t launch_kv_append(const AppendParams& p, cudaStream_t stream)
{
    if (p.total_rows <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((p.total_rows + kAppendWarps - 1) / kAppendWarps));
    cfg.blockDim = dim3(kAppendWarps * 32);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (p.k_scale != nullptr) return launch_append_d<128, true>(p, cfg);
    return p.D == 128 ? launch_append_d<128, false>(p, cfg) : launch_append_d<64, false>(p, cfg);
}

}  // namespace cf

namespace cf {

// fp8 cache, prefill path: one CTA per (page of a prefill sequence, KV head) expands the page's 16 x 128 e4m3 codes
// of K and of V into bf16 (exactly: every e4m3 value is a bf16 value; the per-head scales are applied later, in fp32)
// at the page's place in the staging pools, laid out [stage page, Hkv, 16, 128]; the CTA of head 0 also writes the
// staging block-table entry.  Pages left of a sliding window are not listed and never touched.
__global__ void __launch_bounds__(128) kv_dequant_gather_kernel(const AttnParams p, const __grid_constant__ PlanBytes<kSmallPlanBytes> inl,
                                                                 __nv_bfloat16* __restrict__ stage_k, __nv_bfloat16* __restrict__ stage_v,
                                                                 int32_t* __restrict__ stage_table)
{
    const StageSeq sq = plan_list<StageSeq>(p.plan.base != nullptr ? p.plan.base : inl.bytes, p.plan.stage)[blockIdx.y];
    const int pg = blockIdx.x / p.Hkv, g = blockIdx.x % p.Hkv;
    if (pg >= sq.n_pages) return;
    int32_t blk = __ldg(p.block_table + (int64_t)sq.seq * p.max_blocks + sq.page0 + pg);
    if ((uint32_t)blk >= (uint32_t)p.num_blocks) {          // never dereferenced: page 0 stands in, the error word says so
        if (threadIdx.x == 0 && p.err) atomicOr(p.err, kErrBlockId);
        blk = 0;
    }
    const int spage = sq.stage_base + pg;
    if (g == 0 && threadIdx.x == 0) stage_table[(int64_t)sq.seq * p.max_blocks + sq.page0 + pg] = spage;
    const uint8_t* k8 = reinterpret_cast<const uint8_t*>(p.k_cache) + (int64_t)blk * p.ks_block + (int64_t)g * p.ks_head;
    const uint8_t* v8 = reinterpret_cast<const uint8_t*>(p.v_cache) + (int64_t)blk * p.vs_block + (int64_t)g * p.vs_head;
    // 16 tokens x 8 chunks of 16 codes = 128 chunks per tensor: one per thread
    const int t = threadIdx.x >> 3, c = threadIdx.x & 7;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        const uint4 in = __ldg(reinterpret_cast<const uint4*>((which ? v8 + t * p.vs_token : k8 + t * p.ks_token) + c * 16));
        const uint32_t w[4] = {in.x, in.y, in.z, in.w};
        uint32_t out[8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t f16x2;
                const uint16_t two = (uint16_t)(w[i] >> (16 * h));
                asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(f16x2) : "h"(two));
                const float2 f = __half22float2(*reinterpret_cast<__half2*>(&f16x2));
                out[2 * i + h] = pack_bf16(f.x, f.y);
            }
        __nv_bfloat16* dst = (which ? stage_v : stage_k) + (((int64_t)spage * p.Hkv + g) * 16 + t) * 128 + c * 16;
        *reinterpret_cast<uint4*>(dst) = make_uint4(out[0], out[1], out[2], out[3]);
        *(reinterpret_cast<uint4*>(dst) + 1) = make_uint4(out[4], out[5], out[6], out[7]);
    }
}

cudaError_t launch_kv_dequant_gather(const AttnParams& p, const HostPlan& hp, int n_seqs, int max_pages,
                                     __nv_bfloat16* stage_k, __nv_bfloat16* stage_v, int32_t* stage_table, cudaStream_t stream)
{
    if (n_seqs <= 0 || max_pages <= 0) return cudaSuccess;
    dim3 grid((unsigned)(max_pages * p.Hkv), (unsigned)n_seqs);
    PlanBytes<kSmallPlanBytes> inl;
    if (hp.bytes) std::memcpy(inl.bytes, hp.bytes, hp.size);
    kv_dequant_gather_kernel<<<grid, 128, 0, stream>>>(p, inl, stage_k, stage_v, stage_table);
    return cudaGetLastError();
}

}  // namespace cf
