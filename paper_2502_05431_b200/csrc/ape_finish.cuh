// The end of a row, shared by the merge kernel and by the kernels that merge inside a thread-block cluster: from the row's two
// segments (context and non-context: running maximum M in base-2 units, sum of weights L, unnormalised output acc) to the stored
// result.  A row belongs to a warp (lane l: elements l VEC .. + VEC) or to eight lanes of one (lane l: elements 4 l .. + 4 of every 32).
#pragma once

#include "ape_common.cuh"
#include "ape_kernels.h"

namespace ape {

constexpr float kLn2 = 0.6931471805599453f;

// The end of Eq. 5 for one row, in base-2 units: lse_c already carries S; the segments' sums of weights (norm_*) and of weighted
// values (ac, ao) still carry their own normalisers.
template <int VEC, int LANES = 32>
__device__ __forceinline__ void write_row(const RowsOut& p, int64_t out_row, int h, int lane, float lse_c, float norm_c,
                                          const float (&ac)[VEC], float lse_o, float norm_o, const float (&ao)[VEC])
{
    const float top = fmaxf(lse_c, lse_o);
    float wc = 0.f, wo = 0.f, sum = 0.f;
    if (top > -INFINITY) {
        const float ec = fast_exp2(lse_c - top), eo = fast_exp2(lse_o - top);
        sum = ec + eo;
        wc = (norm_c > 0.f) ? ec / (norm_c * sum) : 0.f;      // weight of the context segment over its own normaliser
        wo = (norm_o > 0.f) ? eo / (norm_o * sum) : 0.f;
    }
    __nv_bfloat16* dst = p.out.data + out_row * p.out.token_stride + static_cast<int64_t>(h) * p.out.head_stride + lane * (LANES == 32 ? VEC : 4);
    float r[VEC];
    #pragma unroll
    for (int v = 0; v < VEC; ++v) r[v] = wc * ac[v] + wo * ao[v];
    if constexpr (LANES != 32) {
        #pragma unroll
        for (int v = 0; v < VEC; v += 4) {
            uint2 pk; pk.x = pack_bf16x2(r[v], r[v + 1]); pk.y = pack_bf16x2(r[v + 2], r[v + 3]);
            *reinterpret_cast<uint2*>(dst + v * LANES) = pk;
        }
    } else if constexpr (VEC == 4) {
        uint2 pk; pk.x = pack_bf16x2(r[0], r[1]); pk.y = pack_bf16x2(r[2], r[3]);
        *reinterpret_cast<uint2*>(dst) = pk;
    } else {
        *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(r[0], r[1]);
    }
    if (p.lse_out != nullptr && lane == 0) p.lse_out[out_row * p.H_q + h] = (top > -INFINITY) ? (top + fast_log2(sum)) * kLn2 : -INFINITY;
}

// Index 0: context, 1: non-context.
template <int VEC, int LANES = 32>
__device__ __forceinline__ void finish_row(const RowsOut& p, int64_t out_row, int h, int lane, const float (&M)[2], const float (&L)[2],
                                           const float (&acc)[2][VEC])
{
    if (p.part_o_ctx != nullptr) {
        // one shard of a context-sharded attend: hand out the two segments as they are
        const int64_t rh = out_row * p.H_q + h;
        const float ic = (L[0] > 0.f) ? 1.f / L[0] : 0.f, io = (L[1] > 0.f) ? 1.f / L[1] : 0.f;
        #pragma unroll
        for (int v = 0; v < VEC; ++v) {
            const int e = (LANES == 32) ? lane * VEC + v : (v / 4 * LANES + lane) * 4 + v % 4;
            p.part_o_ctx[rh * (VEC * LANES) + e] = acc[0][v] * ic;
            p.part_o_oth[rh * (VEC * LANES) + e] = acc[1][v] * io;
        }
        if (lane == 0) {
            p.part_lse_ctx[rh] = (L[0] > 0.f) ? (M[0] + fast_log2(L[0])) * kLn2 : -INFINITY;
            p.part_lse_oth[rh] = (L[1] > 0.f) ? (M[1] + fast_log2(L[1])) * kLn2 : -INFINITY;
        }
        return;
    }
    // base-2 log-sum-exp of the context segment, multiplied by S (Eq. 5: Z_C^S)
    const float lse_c = (L[0] > 0.f) ? p.S * (M[0] + fast_log2(L[0])) : -INFINITY;
    const float lse_o = (L[1] > 0.f) ? (M[1] + fast_log2(L[1])) : -INFINITY;
    write_row<VEC, LANES>(p, out_row, h, lane, lse_c, L[0], acc[0], lse_o, L[1], acc[1]);
}

// ---- thread-block clusters -------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
// All threads of all blocks of the cluster; what was written before the arrival is visible behind the wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// The address, in block `rank` of the cluster, of what this block has at smem_addr
__device__ __forceinline__ uint32_t cluster_map(uint32_t smem_addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
    return r;
}
// An arrival that orders no memory: for blocks that only tell each other that they may leave.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_st2(uint32_t addr, float a, float b) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void cluster_st4(uint32_t addr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// Stores and copies to another block's shared memory, counted in bytes on a barrier there: who waits on it (mbar_wait_received) sees them, no barrier
// of the whole cluster is needed.  addr / dst and bar: addresses of the same block (cluster_map).
__device__ __forceinline__ void cluster_send2(uint32_t addr, float a, float b, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_copy(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {       // 16-byte pieces
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}

// One warp merges one row of a cluster whose blocks have each sent at most one partial of it to this block: those of blocks
// [0, n_ctx) belong to the context, those of the n_oth behind them do not.  ml[j]: (m, l) of block j's partial; o + j * stride: this
// lane's VEC elements of it.
template <int VEC>
__device__ __forceinline__ void merge_received(const float2* ml, const float* o, int stride, int n_ctx, int n_oth,
                                               float (&M)[2], float (&L)[2], float (&acc)[2][VEC])
{
    // Every lane reads all (m, l) itself: a chain of two reads, not of twenty shuffles (1,300 cycles).
    #pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
        const int j0 = seg ? n_ctx : 0, j1 = seg ? n_ctx + n_oth : n_ctx;
        float top = -INFINITY;
        #pragma unroll 4
        for (int j = j0; j < j1; ++j) top = fmaxf(top, ml[j].x);
        const float base = (top == -INFINITY) ? 0.f : top;
        float sum = 0.f;
        #pragma unroll
        for (int v = 0; v < VEC; ++v) acc[seg][v] = 0.f;
        #pragma unroll 4
        for (int j = j0; j < j1; ++j) {                    // (an empty partial has m = -inf, l = 0 and a row of zeros)
            const float f = fast_exp2(ml[j].x - base);
            sum += ml[j].y * f;
            float x[VEC];
            if constexpr (VEC == 4) { const float4 t = *reinterpret_cast<const float4*>(o + j * stride); x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w; }
            else { const float2 t = *reinterpret_cast<const float2*>(o + j * stride); x[0] = t.x; x[1] = t.y; }
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[seg][v] += f * x[v];
        }
        M[seg] = top; L[seg] = sum;
    }
}

// Merges one row of a cluster whose blocks have each at most one partial of it: those of blocks [0, n_ctx) belong to the context, those
// of the n_oth behind them do not.  ml[j * ml_stride]: (m, l) of block j's partial; load(j, x): this lane's VEC elements of it.
// Short loops: the code runs once per launch, and instructions that the SM does not hold yet cost more than the loops' latencies (behind
// the rows' arrival, 64 rows over 10 x 256 tokens: 3,700 cycles with all sixteen blocks unrolled, 2,700 this way).
// (An empty partial has m = -inf, l = 0 and a row of zeros.)
template <int VEC, typename Load>
__device__ __forceinline__ void merge_cluster(const float2* ml, int ml_stride, int n_ctx, int n_oth, Load load, float (&M)[2], float (&L)[2], float (&acc)[2][VEC])
{
    const int n = n_ctx + n_oth;
    float mc = -INFINITY, mo = -INFINITY;
    #pragma unroll 2
    for (int j = 0; j < n; ++j) {
        const float m = ml[j * ml_stride].x;
        if (j < n_ctx) mc = fmaxf(mc, m); else mo = fmaxf(mo, m);
    }
    M[0] = mc; M[1] = mo; L[0] = L[1] = 0.f;
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[0][v] = acc[1][v] = 0.f;
    #pragma unroll 1
    for (int seg = 0; seg < 2; ++seg) {
        const int j1 = seg ? n : n_ctx;
        const float top = seg ? mo : mc, base = (top == -INFINITY) ? 0.f : top;
        float sum = 0.f, x[VEC], y[VEC];
        #pragma unroll
        for (int v = 0; v < VEC; ++v) y[v] = 0.f;
        #pragma unroll 2
        for (int j = seg ? n_ctx : 0; j < j1; ++j) {
            const float2 w = ml[j * ml_stride];
            load(j, x);
            const float f = fast_exp2(w.x - base);
            sum += w.y * f;
            #pragma unroll
            for (int v = 0; v < VEC; ++v) y[v] += f * x[v];
        }
        if (seg) {
            L[1] = sum;
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[1][v] = y[v];
        } else {
            L[0] = sum;
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[0][v] = y[v];
        }
    }
}

}  // namespace ape
