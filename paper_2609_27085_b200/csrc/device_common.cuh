// Device-side helpers shared by the attention kernels: kernel parameter block and thin PTX wrappers.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "plan.h"

namespace cf {

// Where a call's work-item lists are: byte offsets from `base`, a device copy of the plan, or (base null) from the bytes
// that the launch itself carries.  A small plan travels in the kernels' parameter space instead of through a pinned
// buffer, a copy and an event: a launch costs 0.3 us more with 4 KB of parameters and 1.3 us more with 12 KB (measured on a
// B200), and the first kernel does not wait for a copy engine.
struct PlanRef {
    const uint8_t* base;
    int32_t dec, comb, sh, shm, pre_tc, pre_comb, stage;
};
constexpr int kSmallPlanBytes = 3968, kMidPlanBytes = 12288;
template <int BYTES>
struct PlanBytes {
    alignas(16) uint8_t bytes[BYTES];
};
template <>
struct PlanBytes<0> {
    static constexpr const uint8_t* bytes = nullptr;
};
template <class T>
__device__ __forceinline__ const T* plan_list(const uint8_t* plan, int32_t offset)
{
    return reinterpret_cast<const T*>(plan + offset);
}
// The plan of a host-side call whose lists the launches carry (bytes null: p.plan.base is set instead).  `bytes` lies in a
// buffer of at least kSmallPlanBytes, for larger plans of kMidPlanBytes: the launches read their parameter from there.
struct HostPlan {
    const uint8_t* bytes = nullptr;
    size_t size = 0;
};

struct AttnParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_cache;
    const __nv_bfloat16* v_cache;
    __nv_bfloat16* out;
    float* lse;                       // may be null
    const int32_t* block_table;
    int32_t max_blocks;
    int32_t num_blocks;               // pool size; block ids outside [0, num_blocks) are skipped and reported
    int64_t ks_block, ks_head, ks_token;
    int64_t vs_block, vs_head, vs_token;
    int32_t Hq, Hkv, G;
    float scale_log2;                 // softmax_scale * log2(e)
    int32_t window;                   // sliding window in tokens (0 = none): row at position p sees keys (p - window, p]
    const float* sinks;               // [Hq] per-head sink logits (natural-log units) or null
    const float* k_scale;             // fp8 cache: [Hkv] dequantisation scales (null: bf16 cache, or scale 1)
    const float* v_scale;
    PlanRef plan;                     // work-item lists of the call
    float* part_o;                    // [slot, Hq, D] fp32 un-normalised partial outputs
    float* part_ml;                   // [slot, Hq, 2] running max (log2 domain) and sum
    int32_t dec_chained;              // the decode grid runs beside the prefill grid before it in the stream (spatial sequence)
    uint32_t* dec_counters;           // [first slot of a split sequence, Hkv] chunks finished; null: the combine kernel merges
    float* pre_part_o;                // [row slot, D] fp32 partial rows of KV-split prefill items
    float* pre_part_ml;               // [row slot, 2]
    uint32_t* pre_queue;              // [2] ticket counter of the persistent prefill CTAs, and how many of them have left
    uint32_t* err;                    // device error word (bits below); may be null
};

// Start of a decode grid.  Every decode kernel is launched with programmatic stream serialisation.  On its own it waits
// for the grid before it in the stream (the append) before its first read of anything but its work item.  Behind the
// front prefill grid of the spatial sequence (p.dec_chained) it must not wait for that grid, and need not: every CTA of
// the front grid has waited for the append before it allowed this grid to start.  There the grid has one CTA more than
// work, which waits for the front grid, so that completion of this grid implies completion of that one.
__device__ __forceinline__ void decode_grid_start(const AttnParams& p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!p.dec_chained) asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ bool decode_extra_cta(const AttnParams& p)      // true in that extra CTA, once it has waited
{
    if (!p.dec_chained || blockIdx.x != gridDim.x - 1) return false;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return true;
}

// Bits of the device error word
constexpr uint32_t kErrTimeout = 1u;      // a bounded wait expired
constexpr uint32_t kErrBlockId = 2u;      // a block-table entry in use lay outside the pool; its page was skipped

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte async copy global -> shared, L2 only; src_bytes = 0 zero-fills the destination.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// The same with an L2 eviction policy (createpolicy): K/V pages that decode streams once are marked
// evict-first, so that they do not push the prefill kernel's re-read K/V tiles out of L2.
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void cp_async16_hint(uint32_t dst, const void* src, int src_bytes, uint64_t policy)
{
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;\n" ::"r"(dst), "l"(src), "r"(src_bytes), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// transpose an 8x8 tile of 16-bit values held one row-pair per thread
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a)
{
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
    return d;
}
// D(16x8, f32) += A(16x16, bf16, row) * B(16x8, bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);   // .x = lo (low 16 bits), .y = hi
    return *reinterpret_cast<uint32_t*>(&v);
}

// Byte offset of 16-byte chunk `c` (0..D/8) of token row `t` inside a K/V tile stored as
// [D/64 halves][rows][64 elements] with the 16-byte chunks of every 128-byte row XOR-swizzled by
// the row index, so that 8 consecutive rows at one logical chunk hit 8 different bank groups.
template <int ROWS>
__device__ __forceinline__ uint32_t tile_off(int t, int c)
{
    return (uint32_t)((c >> 3) * (ROWS * 128) + t * 128 + (((c & 7) ^ (t & 7)) << 4));
}

constexpr float kLn2 = 0.6931471805599453f;
constexpr float kLog2e = 1.4426950408889634f;

// Joins a sink logit (log2 domain) to a softmax whose running maximum is M and un-normalised sum is L: the sink
// adds 2^(sink - M') to the sum and carries no value.  Returns the factor by which the un-normalised output
// must shrink (1 when the maximum does not move); M and L are updated.  M may be -inf only together with L = 0.
__device__ __forceinline__ float join_sink(float sink2, float& M, float& L)
{
    const float Mn = fmaxf(M, sink2);
    const float f = fast_exp2(M - Mn);
    L = L * f + fast_exp2(sink2 - Mn);
    M = Mn;
    return f;
}

}  // namespace cf
