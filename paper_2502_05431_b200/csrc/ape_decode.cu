// Split-KV decode kernel of APE attention: one new query token per request streams the whole cached
// sequence [prefix | contexts | query segment] once.  HBM-bound: K/V tiles are brought in by the bulk
// tensor copy engine through a multi-stage shared-memory ring; the small (G heads) x (16 tokens) products run on
// warp-level mma so that arithmetic never limits the stream.  Each work item covers tiles of ONE segment
// (context, or prefix + query segment) and emits one partial (m, l, O~) in base-2 units; the merge kernel
// applies the hierarchical softmax identity and Eq. 5's S afterwards.
#include "ape_common.cuh"
#include "ape_finish.cuh"
#include "ape_kernels.h"

namespace ape {

namespace {

constexpr int kTile = kDecodeTile;          // tokens per stage
constexpr int kGroups = 2;                  // of four warps; warp w belongs to group w / 4, which takes every other tile
constexpr int kConsumerWarps = 4 * kGroups;
constexpr int kThreads = (kConsumerWarps + 1) * 32;
// Tile n is group n % kGroups's and lies in stage n % depth, and the depth is a multiple of kGroups, so that a stage always belongs to the
// same group.  A wait tells the phases of a barrier apart by their parity only: a group that saw every other use of a stage could take a
// phase that has not ended for the one before it, and read a tile that is still landing.
constexpr int kMaxStages = 8;
static_assert(kMaxStages % kGroups == 0);
constexpr int kRecvRows = 32;               // (m, l) of a block's share of the rows, from every block: G, at most 16, rounded up to a multiple of the size
constexpr bool shares_fit() {
    for (int c : kCluster)
        for (int G = 1; G <= 16; ++G)
            if ((G + c - 1) / c * c > kRecvRows) return false;
    return true;
}
static_assert(shares_fit(), "a block's share of the rows does not fit");

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Byte offset of 16-byte chunk `chunk` (0 .. D/8-1) of token row `row` inside a K or V stage that the copy engine
// wrote as D/64 slabs of [kTile rows][128 B] with the 128-byte swizzle.
__device__ __forceinline__ uint32_t swz(int row, int chunk) {
    return static_cast<uint32_t>((chunk >> 3) * (kTile * 128) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
}

// 8 x 8 b16 matrix across the warp (lane: two elements of row lane / 4), transposed
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}

// The products of a warp with a slice of 16 tokens of a tile, and its running partial (m, l, O~) of the G query heads.  Two forms:
//
// HeadsAsColumns, at most eight heads: S^T = K Q^T and O^T = V^T P^T, so the tokens (or the elements of a head) are the 16 rows of an mma
// and the heads its 8 columns, half the products that 16 rows for the heads take (of which four heads use a quarter).  A step that is not
// bound by HBM is bound by these chains, in a graph of calls: 4 requests over 4 x 256 tokens 6.05 -> 5.74 us, 8 over 50 x 256 tokens (two KV heads of 64)
// 13.4 -> 12.5, 4 over 100 x 256 (eight KV heads of one query head) 69.9 -> 68.2; 16 over 500 x 256, at the HBM rate, as before.
// HeadsAsRows, 16 heads: O = P V with the heads as the rows.  As columns they are two groups, so as many products, and the maxima over the
// tokens take three shuffles a head instead of two: 4 requests over 30 x 256 tokens 8.5 us, as columns 8.9.
template <int D>
struct HeadsAsColumns {
    static constexpr int kKSteps = D / 16;
    static constexpr int kRow = D + 4;      // floats between rows of the partials: a store of 8 elements of every second row falls on 32 banks
    uint32_t qb[kKSteps][2];        // Q^T (D x 8; columns >= G are zero)
    float o[D / 16][4];             // O^T: element 16 j + qr (+ 8) of heads 2 qc, + 1; m and l are those heads'
    float m[2], l[2];

    // Plain loads of Q: this grid exists while the kernel before it, which may be writing Q, still runs, and the read-only path is for data
    // that nobody writes in a grid's lifetime.
    __device__ __forceinline__ void begin(const __nv_bfloat16* q, int64_t head_stride, int G) {
        const int lane = threadIdx.x & 31, qr = lane >> 2, qc = lane & 3;
        #pragma unroll
        for (int ks = 0; ks < kKSteps; ++ks) {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(q + qr * head_stride + ks * 16 + 2 * qc);
            qb[ks][0] = (qr < G) ? src[0] : 0u;
            qb[ks][1] = (qr < G) ? src[4] : 0u;
        }
        #pragma unroll
        for (int j = 0; j < D / 16; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
        m[0] = m[1] = -INFINITY; l[0] = l[1] = 0.f;
    }

    __device__ __forceinline__ void tile(uint32_t k_s, uint32_t v_s, int tok0, int n_valid, float scale) {
        const int lane = threadIdx.x & 31, qr = lane >> 2;
        // (even and odd steps of the head dimension in accumulators of their own: half the chain of dependent products)
        float sc[4] = {0.f, 0.f, 0.f, 0.f}, sd[4] = {0.f, 0.f, 0.f, 0.f};
        {
            const int row = tok0 + (lane & 15), chunk_sel = lane >> 4;
            #pragma unroll
            for (int ks = 0; ks < kKSteps; ++ks) {
                uint32_t a[4];
                ldmatrix_x4(k_s + swz(row, 2 * ks + chunk_sel), a[0], a[1], a[2], a[3]);
                mma_bf16_16816((ks & 1) ? sd : sc, a, qb[ks][0], qb[ks][1]);
            }
        }
        // base-2 logits of this lane's two tokens and two heads, validity mask
        const bool v0 = tok0 + qr < n_valid, v1 = tok0 + qr + 8 < n_valid;
        float x[4];
        #pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = (i < 2 ? v0 : v1) ? (sc[i] + sd[i]) * scale : -INFINITY;
        float mx0 = fmaxf(x[0], x[2]), mx1 = fmaxf(x[1], x[3]);
        #pragma unroll
        for (int d = 4; d < 32; d *= 2) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, d));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, d));
        }
        const float mn0 = fmaxf(m[0], mx0), mn1 = fmaxf(m[1], mx1);       // finite: the slice holds a valid key
        if (__any_sync(0xffffffffu, (mn0 > m[0]) | (mn1 > m[1]))) {
            const float f0 = fast_exp2(m[0] - mn0), f1 = fast_exp2(m[1] - mn1);
            l[0] *= f0; l[1] *= f1;
            #pragma unroll
            for (int j = 0; j < D / 16; ++j) { o[j][0] *= f0; o[j][1] *= f1; o[j][2] *= f0; o[j][3] *= f1; }
            m[0] = mn0; m[1] = mn1;
        }
        const float p0 = fast_exp2(x[0] - m[0]), p1 = fast_exp2(x[1] - m[1]), p2 = fast_exp2(x[2] - m[0]), p3 = fast_exp2(x[3] - m[1]);
        l[0] += p0 + p2;
        l[1] += p1 + p3;
        const uint32_t b0 = movmatrix_trans(pack_bf16x2(p0, p1)), b1 = movmatrix_trans(pack_bf16x2(p2, p3));
        {
            const int row = tok0 + ((lane >> 4) << 3) + (lane & 7), chunk_sel = (lane >> 3) & 1;
            #pragma unroll
            for (int j = 0; j < D / 16; ++j) {
                uint32_t a[4];
                ldmatrix_x4_trans(v_s + swz(row, 2 * j + chunk_sel), a[0], a[1], a[2], a[3]);
                mma_bf16_16816(o[j], a, b0, b1);
            }
        }
    }

    // into shared memory: row g at rows + g * RS, its (m, l) at ms[8 g], ls[8 g]
    __device__ __forceinline__ void hand_in(float* rows, float* ms, float* ls, int G) {
        constexpr int RS = kRow;
        const int lane = threadIdx.x & 31, qr = lane >> 2, qc = lane & 3;
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = 2 * qc + h;
            #pragma unroll
            for (int d = 4; d < 32; d *= 2) l[h] += __shfl_xor_sync(0xffffffffu, l[h], d);
            if (qr == 0) { ms[row * 8] = m[h]; ls[row * 8] = l[h]; }
            if (row < G) {
                float* dst = rows + row * RS + qr;
                #pragma unroll
                for (int j = 0; j < D / 16; ++j) { dst[16 * j] = o[j][h]; dst[16 * j + 8] = o[j][2 + h]; }
            }
        }
    }
};

template <int D>
struct HeadsAsRows {
    static constexpr int kKSteps = D / 16;
    static constexpr int kRow = D + 8;      // (pairs of elements of eight rows)
    uint32_t qa[kKSteps][4];        // Q (16 x D; rows >= G are zero)
    float o[D / 8][4];              // O: heads qr, qr + 8, elements 8 j + 2 qc, + 1
    float m_lo, m_hi, l_lo, l_hi;

    __device__ __forceinline__ void begin(const __nv_bfloat16* q, int64_t head_stride, int G) {
        const int lane = threadIdx.x & 31, qr = lane >> 2, qc = lane & 3;
        #pragma unroll
        for (int ks = 0; ks < kKSteps; ++ks) {
            const uint32_t* r_lo = reinterpret_cast<const uint32_t*>(q + qr * head_stride + ks * 16 + 2 * qc);
            const uint32_t* r_hi = reinterpret_cast<const uint32_t*>(q + (qr + 8) * head_stride + ks * 16 + 2 * qc);
            qa[ks][0] = (qr < G) ? *r_lo : 0u;
            qa[ks][1] = (qr + 8 < G) ? *r_hi : 0u;
            qa[ks][2] = (qr < G) ? r_lo[4] : 0u;
            qa[ks][3] = (qr + 8 < G) ? r_hi[4] : 0u;
        }
        #pragma unroll
        for (int j = 0; j < D / 8; ++j) { o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f; }
        m_lo = m_hi = -INFINITY; l_lo = l_hi = 0.f;
    }

    __device__ __forceinline__ void tile(uint32_t k_s, uint32_t v_s, int tok0, int n_valid, float scale) {
        const int lane = threadIdx.x & 31, qc = lane & 3;
        // S = Q K^T for 16 tokens: two n-tiles of 8 tokens
        // (even and odd steps of the head dimension in accumulators of their own: half the chain of dependent products)
        float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}}, sd[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        {
            const int row = tok0 + ((lane >> 4) << 3) + (lane & 7);
            const int chunk_sel = (lane >> 3) & 1;
            #pragma unroll
            for (int ks = 0; ks < kKSteps; ++ks) {
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4(k_s + swz(row, 2 * ks + chunk_sel), b0, b1, b2, b3);
                mma_bf16_16816((ks & 1) ? sd[0] : sc[0], qa[ks], b0, b1);
                mma_bf16_16816((ks & 1) ? sd[1] : sc[1], qa[ks], b2, b3);
            }
            #pragma unroll
            for (int i = 0; i < 4; ++i) { sc[0][i] += sd[0][i]; sc[1][i] += sd[1][i]; }
        }
        // base-2 logits, validity mask
        #pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const int c0 = tok0 + nt * 8 + 2 * qc;
            const bool v0 = c0 < n_valid, v1 = c0 + 1 < n_valid;
            sc[nt][0] = v0 ? sc[nt][0] * scale : -INFINITY;
            sc[nt][1] = v1 ? sc[nt][1] * scale : -INFINITY;
            sc[nt][2] = v0 ? sc[nt][2] * scale : -INFINITY;
            sc[nt][3] = v1 ? sc[nt][3] * scale : -INFINITY;
        }
        float mx_lo = fmaxf(fmaxf(sc[0][0], sc[0][1]), fmaxf(sc[1][0], sc[1][1]));
        float mx_hi = fmaxf(fmaxf(sc[0][2], sc[0][3]), fmaxf(sc[1][2], sc[1][3]));
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
        mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
        mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
        const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);   // finite: the slice holds a valid key
        if (__any_sync(0xffffffffu, (mn_lo > m_lo) | (mn_hi > m_hi))) {
            const float f_lo = fast_exp2(m_lo - mn_lo), f_hi = fast_exp2(m_hi - mn_hi);
            l_lo *= f_lo; l_hi *= f_hi;
            #pragma unroll
            for (int j = 0; j < D / 8; ++j) { o[j][0] *= f_lo; o[j][1] *= f_lo; o[j][2] *= f_hi; o[j][3] *= f_hi; }
            m_lo = mn_lo; m_hi = mn_hi;
        }
        uint32_t pa[4];
        {
            const float p00 = fast_exp2(sc[0][0] - m_lo), p01 = fast_exp2(sc[0][1] - m_lo);
            const float p02 = fast_exp2(sc[0][2] - m_hi), p03 = fast_exp2(sc[0][3] - m_hi);
            const float p10 = fast_exp2(sc[1][0] - m_lo), p11 = fast_exp2(sc[1][1] - m_lo);
            const float p12 = fast_exp2(sc[1][2] - m_hi), p13 = fast_exp2(sc[1][3] - m_hi);
            l_lo += (p00 + p01) + (p10 + p11);
            l_hi += (p02 + p03) + (p12 + p13);
            pa[0] = pack_bf16x2(p00, p01); pa[1] = pack_bf16x2(p02, p03);
            pa[2] = pack_bf16x2(p10, p11); pa[3] = pack_bf16x2(p12, p13);
        }
        // O += P V
        {
            const int row = tok0 + (((lane >> 3) & 1) << 3) + (lane & 7);
            const int chunk_sel = lane >> 4;
            #pragma unroll
            for (int j = 0; j < D / 16; ++j) {
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4_trans(v_s + swz(row, 2 * j + chunk_sel), b0, b1, b2, b3);
                mma_bf16_16816(o[2 * j], pa, b0, b1);
                mma_bf16_16816(o[2 * j + 1], pa, b2, b3);
            }
        }
    }

    __device__ __forceinline__ void hand_in(float* rows, float* ms, float* ls, int G) {
        constexpr int RS = kRow;
        const int lane = threadIdx.x & 31, qr = lane >> 2, qc = lane & 3;
        l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1); l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
        l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1); l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
        if (qc == 0) {
            ms[qr * 8] = m_lo; ms[(qr + 8) * 8] = m_hi;
            ls[qr * 8] = l_lo; ls[(qr + 8) * 8] = l_hi;
        }
        #pragma unroll
        for (int j = 0; j < D / 8; ++j) {
            const int e = j * 8 + 2 * qc;
            if (qr < G) *reinterpret_cast<float2*>(&rows[qr * RS + e]) = make_float2(o[j][0], o[j][1]);
            if (qr + 8 < G) *reinterpret_cast<float2*>(&rows[(qr + 8) * RS + e]) = make_float2(o[j][2], o[j][3]);
        }
    }
};

}  // namespace

// A long step is bound by HBM (16 requests over 128K tokens: 6.7 TB/s), a short one by a chain of latencies, in cycles for one request
// over 10 x 256 tokens: wait for the kernel before -> first tile 1,500 (2,200 when the records and the copy engine's descriptors
// are fetched behind that wait), 950 per tile of a warp, 750 for the partials of the eight warps (1,430 with a row's (m, l) read one by
// one and rows 128 floats apart), then the merge.  All of them together, in two kernels: 7.4 us per call, then 6.3 to 6.5.
//
// CLUSTER: the blocks of a thread-block cluster share the tiles of one (request, KV head), one item each, and merge their partials
// themselves: each block sends the rows of its partial to the blocks that merge them (distributed shared memory, one barrier of the
// cluster), so that a short step is one kernel, no partial goes to memory and no second kernel waits for the last block of the
// first: 5.9 us for the step above, and in a graph of calls 3.6 instead of 4.7 for a single context of 64 tokens.  (Sent, not fetched: reading the others'
// partials behind the barrier cost another 1,600 cycles and a second barrier before a block may leave.)
template <int D, bool CLUSTER, typename Products>
__global__ void __launch_bounds__(kThreads, 1)
ape_decode_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                  const __grid_constant__ DecodeParams p)
{
    constexpr int kSlabs = D / 64;
    constexpr int kStageBytes = 2 * kTile * D * 2;      // K + V

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int n_stages = p.n_stages;
    uint8_t* stage_base = smem;
    constexpr int RS = Products::kRow;
    float* red = reinterpret_cast<float*>(smem + static_cast<size_t>(n_stages) * kStageBytes);  // [8][G][RS], then [16][8] m, [16][8] l
    float* red_m = red + kConsumerWarps * p.G * RS;
    float* red_l = red_m + kConsumerWarps * 16;
    uint64_t* bars = reinterpret_cast<uint64_t*>(red_l + kConsumerWarps * 16);   // full[n_stages], empty[n_stages]
    __shared__ int abort_flag;
    __shared__ int stage_valid[kMaxStages];              // keys of the tile in a stage that count
    // CLUSTER: what the blocks of the cluster send this one, row r of the group to block r mod cluster: at index (r / cluster) * cluster +
    // sender, (m, l) here and the row behind the barriers
    __shared__ float2 recv_ml[kRecvRows];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* recv = reinterpret_cast<float*>(bars + 2 * kMaxStages);
    if (CLUSTER) cluster_arrive();                       // this block's shared memory may be written by the others (they wait for it below)
    const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + n_stages);

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 4);       // one arrival per warp of the group that consumed the stage
        }
        mbar_fence_init();
    }
    // The records (range and item, merge group) are read, and the copy engine's descriptors are fetched, while the kernel before this one
    // ends.  A cluster's blocks find theirs by their index: where clusters cannot be placed before that kernel has left its SMs, a record
    // that is found through another one is 700 cycles more between the two (4 requests over 4 x 256 tokens 6.20 us, now 6.05).
    const int item_begin = CLUSTER ? static_cast<int>(blockIdx.x) : p.cta_item_begin[blockIdx.x];
    DevItem first{};
    int item_end;
    if (CLUSTER) {
        first = p.items[item_begin];
        item_end = item_begin + (first.n_sib > 0 ? 1 : 0);
    } else {
        item_end = p.cta_item_begin[blockIdx.x + 1];
        if (item_begin < item_end) first = p.items[item_begin];
    }
    if (warp == kConsumerWarps && lane == 0) {
        tma_prefetch_desc(&tm_k);
        tma_prefetch_desc(&tm_v);
    }
    DevMerge group{};
    if (CLUSTER) group = p.groups[blockIdx.x / static_cast<unsigned>(p.cluster)];
    // where elements e .. e + 3 of this block's partial of a row go: in the block that merges the row
    auto sent_to = [&](int row) { const int turn = row / p.cluster; return make_int2(row - turn * p.cluster, turn * p.cluster + static_cast<int>(cluster_ctarank())); };
    const int2 first_to = CLUSTER ? sent_to(threadIdx.x / (D / 4)) : make_int2(0, 0);
    // Tiles of an item that this step reads: what the query segment has not grown into yet is left out.
    auto live_end = [&](const DevItem& item) {
        return item.seg == SEG_CTX ? item.tile_end : min(item.tile_end, item.row_block + (item.l_k + p.kv_extra + kTile - 1) / kTile);
    };
    __syncthreads();
    if (CLUSTER) cluster_wait();
    pdl_wait();
    if (p.let_next_in != 0) pdl_trigger();

    if (warp == kConsumerWarps) {
        // ---------------- producer: one lane feeds the ring --------------------------------------------------------
        if (lane == 0) {
            uint32_t cnt = 0;
            bool ok = true;
            for (int it = item_begin; it < item_end && ok; ++it) {
                const DevItem item = (it == item_begin) ? first : p.items[it];
                const int t_end = live_end(item), l_k_now = item.l_k + p.kv_extra;
                for (int t = item.tile_begin; t < t_end; ++t, ++cnt) {
                    const DevTile tile = (t == item.tile_begin) ? item.first_tile : p.tiles[t];
                    const int s = cnt % n_stages;
                    const uint32_t use = cnt / n_stages;
                    if (use > 0 && !mbar_wait(bar_empty + 8 * s, (use & 1) ^ 1, &abort_flag, p.status)) { ok = false; break; }
                    const int tok = tile.tok;
                    stage_valid[s] = (tile.flags & TILE_GROWS) ? min(l_k_now - tile.key_base, kTile) : tile.n_valid;   // (published by the arrival below)
                    const uint32_t dst = smem_u32(stage_base + static_cast<size_t>(s) * kStageBytes);
                    mbar_expect_tx(bar_full + 8 * s, kStageBytes);
                    #pragma unroll
                    for (int sl = 0; sl < kSlabs; ++sl) {
                        tma_load_3d(dst + sl * (kTile * 128), &tm_k, bar_full + 8 * s, sl * 64, item.kv_head, tok);
                        tma_load_3d(dst + kTile * D * 2 + sl * (kTile * 128), &tm_v, bar_full + 8 * s, sl * 64, item.kv_head, tok);
                    }
                }
            }
            // Nothing may still be landing in shared memory when the CTA exits: on an abort, wait (bounded) for the
            // copies already issued.  In the normal case the consumers have waited on every stage already.
            if (!ok) {
                for (int s = 0; s < n_stages; ++s) {
                    const long long t0 = clock64();
                    const uint32_t issued = (cnt > static_cast<uint32_t>(s)) ? (cnt - 1 - s) / n_stages + 1 : 0;
                    if (issued == 0) continue;
                    while (!mbar_try_wait(bar_full + 8 * s, (issued - 1) & 1) && clock64() - t0 < (1ll << 24)) {}
                }
            }
        }
    } else {
        // ---------------- consumers ----------------------------------------------------------------------------------
        const int grp = warp >> 2;
        const int w4 = warp & 3;              // 16-token slice inside a tile
        const int G = p.G;
        uint32_t cnt = 0;

        for (int it = item_begin; it < item_end; ++it) {
            const DevItem item = (it == item_begin) ? first : p.items[it];
            const float scale = (item.seg == SEG_CTX) ? p.scale_ctx_log2 : p.scale_oth_log2;
            const int t_end = live_end(item);

            Products part;
            part.begin(p.q.data + static_cast<int64_t>(item.q_row0) * p.q.token_stride + static_cast<int64_t>(item.kv_head) * G * p.q.head_stride, p.q.head_stride, G);

            for (int t = item.tile_begin; t < t_end; ++t, ++cnt) {
                if (cnt % kGroups != static_cast<uint32_t>(grp)) continue;
                const int s = cnt % n_stages;
                const uint32_t use = cnt / n_stages;
                if (!mbar_wait(bar_full + 8 * s, use & 1, &abort_flag, p.status)) break;
                const int n_valid = stage_valid[s];

                const int tok0 = w4 * 16;
                if (tok0 < n_valid) {
                    const uint32_t k_s = smem_u32(stage_base + static_cast<size_t>(s) * kStageBytes);
                    const uint32_t v_s = k_s + kTile * D * 2;

                    if (n_valid < tok0 + 16) {
                        // ragged tile: V rows past the span may hold anything (even NaN); zero them so that 0 * v stays 0
                        const int row = tok0 + (lane >> 1);
                        if (row >= n_valid) {
                            uint8_t* vrow = stage_base + static_cast<size_t>(s) * kStageBytes + kTile * D * 2;
                            #pragma unroll
                            for (int sl = 0; sl < kSlabs; ++sl) {
                                uint4* dst = reinterpret_cast<uint4*>(vrow + sl * (kTile * 128) + row * 128 + (lane & 1) * 64);
                                dst[0] = dst[1] = dst[2] = dst[3] = make_uint4(0, 0, 0, 0);
                            }
                            fence_proxy_async_smem();   // these generic writes precede the next bulk copy into the stage
                        }
                        __syncwarp();
                    }

                    part.tile(k_s, v_s, tok0, n_valid, scale);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty + 8 * s);
            }

            // ---- combine the eight warps' partials of this item and write one (m, l, O~) to the workspace ------------
            part.hand_in(red + warp * G * RS, red_m + warp, red_l + warp, G);
            // Every consumer warp reaches this barrier, also one that gave up on a wait, so the decision to stop is
            // taken by all of them together.
            named_bar_sync(1, kConsumerWarps * 32);
            if (abort_flag) break;
            // a thread takes four elements of a row: 16-byte reads, the row's eight (m, l) in four of them
            #pragma unroll 1
            for (int idx = threadIdx.x; idx < G * (D / 4); idx += kConsumerWarps * 32) {
                const int row = idx / (D / 4), e = (idx - row * (D / 4)) * 4;
                float f[kConsumerWarps], l[kConsumerWarps];
                #pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 a = *reinterpret_cast<const float4*>(&red_m[row * 8 + 4 * h]), b = *reinterpret_cast<const float4*>(&red_l[row * 8 + 4 * h]);
                    f[4 * h] = a.x; f[4 * h + 1] = a.y; f[4 * h + 2] = a.z; f[4 * h + 3] = a.w;
                    l[4 * h] = b.x; l[4 * h + 1] = b.y; l[4 * h + 2] = b.z; l[4 * h + 3] = b.w;
                }
                float4 x[kConsumerWarps];
                #pragma unroll
                for (int w = 0; w < kConsumerWarps; ++w) x[w] = *reinterpret_cast<const float4*>(&red[(w * G + row) * RS + e]);
                float M = f[0];
                #pragma unroll
                for (int w = 1; w < kConsumerWarps; ++w) M = fmaxf(M, f[w]);
                const float Ms = (M == -INFINITY) ? 0.f : M;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                float L = 0.f;
                #pragma unroll
                for (int w = 0; w < kConsumerWarps; ++w) {
                    const float fw = fast_exp2(f[w] - Ms);
                    acc.x += fw * x[w].x; acc.y += fw * x[w].y; acc.z += fw * x[w].z; acc.w += fw * x[w].w;
                    L += fw * l[w];
                }
                if (CLUSTER) {
                    // a sum that is no positive number: empty, as the merge kernel sees it
                    const bool live = L > 0.f;
                    M = live ? M : -INFINITY; L = live ? L : 0.f;
                    acc.x = live ? acc.x : 0.f; acc.y = live ? acc.y : 0.f; acc.z = live ? acc.z : 0.f; acc.w = live ? acc.w : 0.f;
                    const int2 to = (idx < kConsumerWarps * 32) ? first_to : sent_to(row);
                    cluster_st4(cluster_map(smem_u32(recv + to.y * RS + e), to.x), acc);
                    if (e == 0) cluster_st2(cluster_map(smem_u32(&recv_ml[to.y]), to.x), M, L);
                } else {
                    *reinterpret_cast<float4*>(p.ws_o + (static_cast<size_t>(item.slot) * G + row) * D + e) = acc;
                    if (e == 0) *reinterpret_cast<float2*>(p.ws_ml + (static_cast<size_t>(item.slot) * G + row) * 2) = make_float2(M, L);
                }
            }
            if (it + 1 < item_end) named_bar_sync(1, kConsumerWarps * 32);     // before the next item's partials overwrite these
        }
    }

    if constexpr (CLUSTER) {
        constexpr int VEC = D / 32;
        __syncwarp();
        cluster_arrive();
        cluster_wait();                                  // every block's partials are where they belong; nobody reads another block's memory
        const int C = p.cluster;
        for (int turn = warp, row; (row = static_cast<int>(cluster_ctarank()) + C * turn) < p.G; turn += kThreads / 32) {
            const int at = turn * C;
            float M[2], L[2], acc[2][VEC];
            merge_received<VEC>(&recv_ml[at], recv + at * RS + lane * VEC, RS, group.ctx_n, group.oth_n, M, L, acc);
            finish_row<VEC>(p.fin, first.q_row0, group.kv_head * p.G + row, lane, M, L, acc);
        }
    }
}

size_t decode_smem_bytes(int D, int G, int n_stages, int cluster) {
    const int row = G <= 8 ? HeadsAsColumns<128>::kRow - 128 + D : HeadsAsRows<128>::kRow - 128 + D;
    return 1024 + static_cast<size_t>(n_stages) * (2 * kTile * D * 2)
           + sizeof(float) * (kConsumerWarps * G * row + 2 * kConsumerWarps * 16) + 16 * kMaxStages
           + (cluster > 0 ? sizeof(float) * row * ((G + cluster - 1) / cluster * cluster) : 0);
}

int decode_pick_stages(int D, int G, size_t smem_limit, int cluster) {
    int n = kMaxStages;
    while (n > kGroups && decode_smem_bytes(D, G, n, cluster) > smem_limit) n -= kGroups;
    return decode_smem_bytes(D, G, n, cluster) <= smem_limit ? n : 0;
}

using DecodeKernel = void(CUtensorMap, CUtensorMap, DecodeParams);
template <int D>
static DecodeKernel* decode_kernel(bool cluster, int G) {
    if (G <= 8) return cluster ? ape_decode_kernel<D, true, HeadsAsColumns<D>> : ape_decode_kernel<D, false, HeadsAsColumns<D>>;
    return cluster ? ape_decode_kernel<D, true, HeadsAsRows<D>> : ape_decode_kernel<D, false, HeadsAsRows<D>>;
}
static DecodeKernel* decode_kernel(int D, bool cluster, int G) { return D == 128 ? decode_kernel<128>(cluster, G) : decode_kernel<64>(cluster, G); }

cudaError_t launch_decode(int D, const CUtensorMap& tm_k, const CUtensorMap& tm_v, const DecodeParams& p,
                          int n_cta, size_t smem_bytes, bool early, cudaStream_t stream)
{
    const bool c = p.cluster > 0;
    auto* kernel = decode_kernel(D, c, p.G);
    return c ? launch_cluster(p.cluster, early, kernel, n_cta, kThreads, smem_bytes, stream, tm_k, tm_v, p)
             : launch_kernel(early, kernel, n_cta, kThreads, smem_bytes, stream, tm_k, tm_v, p);
}

cudaError_t decode_set_smem_attr(int D, size_t smem_limit) {
    for (int g : {8, 16})
        for (bool c : {false, true}) {
            auto* kernel = decode_kernel(D, c, g);
            cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem_limit));
            if (e == cudaSuccess && c) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

int decode_max_clusters(int D, int cluster, size_t smem_limit) {
    return max_clusters(cluster, decode_kernel(D, true, 8), kThreads, smem_limit);
}

}  // namespace ape
