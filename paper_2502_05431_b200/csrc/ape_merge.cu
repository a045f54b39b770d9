// Merge kernel: turns the per-item partials (m, l, O~), kept in base-2 units, into the final output.
//   1. inside each segment (context / non-context) the partials of all splits are combined by the
//      hierarchical softmax identity (appendix "Hierarchical Formula for Softmax Attention"):
//      LSE = logsumexp_s(m_s + log2 l_s),  O = sum_s 2^(LSE_s - LSE) O_s;
//   2. the context log-sum-exp is multiplied by the scaling factor S and the two segments are merged by a
//      softmax over [S * LSE_C, LSE_other] (Eq. 5; appendix "Efficient Implementation").
// An output row (query token, query head) belongs to one warp, to eight or to eight lanes of one; lanes cover the head dimension.
#include "ape_common.cuh"
#include "ape_finish.cuh"
#include "ape_kernels.h"

namespace ape {

namespace {

template <int VEC>
__device__ __forceinline__ void combine_segment(const float* ws_o, const float* ws_ml,
                                                int slot0, int n, int stride, int rows_per_slot, int row, int D,
                                                int lane, float& M, float& L, float (&acc)[VEC])
{
    M = -INFINITY; L = 0.f;
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    // The partials are independent of each other: their loads are issued eight at a time, then folded in order (a merge
    // with many partials per row, such as a decode batch that shares its contexts, is bound by the latency of these loads).
    constexpr int kBatch = 8;
    for (int i0 = 0; i0 < n; i0 += kBatch) {
        float2 ml[kBatch];
        float x[kBatch][VEC];
        #pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const size_t slot = static_cast<size_t>(slot0) + static_cast<size_t>(i0 + u) * stride;
            ml[u] = (i0 + u < n) ? *reinterpret_cast<const float2*>(ws_ml + (slot * rows_per_slot + row) * 2) : make_float2(-INFINITY, 0.f);
        }
        #pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const size_t slot = static_cast<size_t>(slot0) + static_cast<size_t>(i0 + u) * stride;
            const float* src = ws_o + (slot * rows_per_slot + row) * D + lane * VEC;
            // Issued without waiting for (m, l): the row of an empty partial was never written, but it lies inside the
            // workspace, and the fold below never looks at what was read from it.
            if (i0 + u < n) {
                if constexpr (VEC == 4) { const float4 t = *reinterpret_cast<const float4*>(src); x[u][0] = t.x; x[u][1] = t.y; x[u][2] = t.z; x[u][3] = t.w; }
                else { const float2 t = *reinterpret_cast<const float2*>(src); x[u][0] = t.x; x[u][1] = t.y; }
            } else {
                #pragma unroll
                for (int v = 0; v < VEC; ++v) x[u][v] = 0.f;
            }
        }
        #pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            if (!(ml[u].y > 0.f)) continue;          // empty partial
            const float Mn = fmaxf(M, ml[u].x);
            const float f_old = fast_exp2(M - Mn), f_new = fast_exp2(ml[u].x - Mn);
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[v] = acc[v] * f_old + x[u][v] * f_new;
            L = L * f_old + ml[u].y * f_new;
            M = Mn;
        }
    }
}

// Partials i0 .. i0 + B - 1 of a row's context segment, all requested at once (the walks below take them one after the other, and one
// read at a time, each waiting for memory, is what they were bound by).  The row of an empty partial was never written, but it lies
// inside the workspace, and no walk looks at it.
// Decode, per-context form, us per call: 2 requests x 25 contexts of 388 tokens 39 -> 28, 4 x 62 contexts of 1,709 tokens 332 -> 286.
template <int VEC, int B>
struct PartialBatch {
    int id[B];                                        // context ordinal or node
    float2 ml[B];
    float x[B][VEC];
    __device__ __forceinline__ void load(const MergeParams& p, const DevMerge& g, int item0, int i0, int row, int lane) {
        #pragma unroll
        for (int u = 0; u < B; ++u) {
            id[u] = 0; ml[u] = make_float2(-INFINITY, 0.f);
            #pragma unroll
            for (int v = 0; v < VEC; ++v) x[u][v] = 0.f;
            if (i0 + u >= g.ctx_n) continue;
            const size_t at = (static_cast<size_t>(g.ctx_slot0) + static_cast<size_t>(i0 + u) * g.slot_stride) * p.rows_per_slot + row;
            id[u] = p.items[item0 + i0 + u].ctx_id;
            ml[u] = *reinterpret_cast<const float2*>(p.ws_ml + at * 2);
            const float* src = p.ws_o + at * p.D + lane * VEC;
            if constexpr (VEC == 4) { const float4 t = *reinterpret_cast<const float4*>(src); x[u][0] = t.x; x[u][1] = t.y; x[u][2] = t.z; x[u][3] = t.w; }
            else { const float2 t = *reinterpret_cast<const float2*>(src); x[u][0] = t.x; x[u][1] = t.y; }
        }
    }
};

// Per-context form (appendix "Hierarchical Formula for APE", Eq. 11-12): every context C_i keeps its own normalised
// output and enters the final softmax with S * LSE_i.  Partials arrive grouped by context (consecutive slots with the same
// context ordinal); the result is the context segment's normalised output `acc` (to be divided by `norm`) and its
// scaled base-2 log weight `lse` = log2 sum_i 2^(S * LSE_i).
template <int VEC>
__device__ __forceinline__ void combine_per_context(const MergeParams& p, const DevMerge& g, int row, int lane,
                                                    float& lse, float& norm, float (&acc)[VEC])
{
    float top = -INFINITY, Z = 0.f;                   // running maximum of S * LSE_i and sum of 2^(S * LSE_i - top)
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    float M = -INFINITY, L = 0.f, a[VEC];
    #pragma unroll
    for (int v = 0; v < VEC; ++v) a[v] = 0.f;
    const int item0 = g.ctx_slot0 / g.slot_stride;
    int cur = (g.ctx_n > 0) ? p.items[item0].ctx_id : 0;
    auto fold = [&]() {                               // close the current context
        if (L > 0.f) {
            const float li = p.S * (M + fast_log2(L));
            const float tn = fmaxf(top, li);
            const float f_old = fast_exp2(top - tn), f_new = fast_exp2(li - tn) / L;
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[v] = acc[v] * f_old + a[v] * f_new;
            Z = Z * f_old + fast_exp2(li - tn);
            top = tn;
        }
        M = -INFINITY; L = 0.f;
        #pragma unroll
        for (int v = 0; v < VEC; ++v) a[v] = 0.f;
    };
    PartialBatch<VEC, 8> b;
    #pragma unroll 1
    for (int i0 = 0; i0 < g.ctx_n; i0 += 8) {
        b.load(p, g, item0, i0, row, lane);
        #pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (i0 + u >= g.ctx_n) break;
            if (b.id[u] != cur) { fold(); cur = b.id[u]; }
            if (!(b.ml[u].y > 0.f)) continue;
            const float Mn = fmaxf(M, b.ml[u].x);
            const float f_old = fast_exp2(M - Mn), f_new = fast_exp2(b.ml[u].x - Mn);
            #pragma unroll
            for (int v = 0; v < VEC; ++v) a[v] = a[v] * f_old + b.x[u][v] * f_new;
            L = L * f_old + b.ml[u].y * f_new;
            M = Mn;
        }
    }
    fold();
    norm = Z;
    lse = (Z > 0.f) ? top + fast_log2(Z) : -INFINITY;
}

// Context trees (appendix "Future Directions" on top of "Hierarchical Formula for APE"): the partials of a row arrive in
// depth-first order of the nodes their tiles belong to (a node's own tokens, then its subtrees).  A stack of accumulators,
// one per open tree level, follows that order: a partial is added to its node's accumulator; when the walk leaves a node,
// the node is finished -- log-sum-exp A_n and normalised output V_n of its members, by the plain hierarchical softmax
// identity -- and handed to its parent's accumulator as one member with log weight S * A_n if the node is marked, A_n
// otherwise.  Level 0 collects the top-level nodes; its content is the context side of the final softmax.
template <int VEC>
__device__ __forceinline__ void combine_tree(const MergeParams& p, const DevMerge& g, int row, int lane,
                                             float& lse, float& norm, float (&acc)[VEC])
{
    float top[kMaxTreeDepth + 1], Z[kMaxTreeDepth + 1], a[kMaxTreeDepth + 1][VEC];
    int node_at[kMaxTreeDepth + 1];
    top[0] = -INFINITY; Z[0] = 0.f; node_at[0] = -1;
    #pragma unroll
    for (int v = 0; v < VEC; ++v) a[0][v] = 0.f;
    int sp = 0;                                       // deepest open level; level k + 1 holds an open node of depth k
    auto add = [&](int lv, float m, float l, const float (&o)[VEC]) {
        const float Mn = fmaxf(top[lv], m);
        const float f_old = fast_exp2(top[lv] - Mn), f_new = fast_exp2(m - Mn);
        #pragma unroll
        for (int v = 0; v < VEC; ++v) a[lv][v] = a[lv][v] * f_old + o[v] * f_new;
        Z[lv] = Z[lv] * f_old + l * f_new;
        top[lv] = Mn;
    };
    auto close = [&](int lv) {                        // finish the node at level lv and hand it to level lv - 1
        if (Z[lv] > 0.f) {
            const float A = top[lv] + fast_log2(Z[lv]);
            const float handed = p.nodes[node_at[lv]].scaled ? p.S * A : A;
            const float inv = 1.f / Z[lv];
            float o[VEC];
            #pragma unroll
            for (int v = 0; v < VEC; ++v) o[v] = a[lv][v] * inv;
            add(lv - 1, handed, 1.f, o);
        }
    };
    auto ancestor = [&](int node, int depth_now, int depth_want) {
        for (; depth_now > depth_want; --depth_now) node = p.nodes[node].parent;
        return node;
    };
    const int item0 = g.ctx_slot0 / g.slot_stride;
    PartialBatch<VEC, 4> b;
    #pragma unroll 1
    for (int i0 = 0; i0 < g.ctx_n; i0 += 4) {
        b.load(p, g, item0, i0, row, lane);
        #pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i0 + u >= g.ctx_n) break;
            const int node = b.id[u];
            const int depth = p.nodes[node].depth;
            // leave every open node that is not on the path from the top level down to `node`
            while (sp > 0 && (sp - 1 > depth || ancestor(node, depth, sp - 1) != node_at[sp])) { close(sp); --sp; }
            // open the rest of that path
            while (sp < depth + 1) {
                ++sp;
                node_at[sp] = ancestor(node, depth, sp - 1);
                top[sp] = -INFINITY; Z[sp] = 0.f;
                #pragma unroll
                for (int v = 0; v < VEC; ++v) a[sp][v] = 0.f;
            }
            if (b.ml[u].y > 0.f) add(sp, b.ml[u].x, b.ml[u].y, b.x[u]);
        }
    }
    while (sp > 0) { close(sp); --sp; }
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = a[0][v];
    norm = Z[0];
    lse = (Z[0] > 0.f) ? top[0] + fast_log2(Z[0]) : -INFINITY;
}

// Eq. 5 form.  W warps (1 or 8) of a block share a row's partials and meet in shared memory.  The kernel is bound by the latency of its
// loads (records -> (m, l) -> rows of O~), so it is built to have many of them in flight: a lane per partial fetches all (m, l)
// of a row at once, the rows of the first kBatch partials are requested together with them, and few registers per thread
// leave room for many warps (127 before, which left 16 warps per SM: 4 x 128 rows over 20K tokens, 27 MB of partials, 30 us).
// The weights 2^(m - M) are then one exponential per lane, and folding a partial is VEC multiply-adds.
template <int VEC, int W>
__global__ void __launch_bounds__(256, 4) ape_merge_kernel(const MergeParams p)
{
    constexpr int kBatch = 4;
    constexpr int D = VEC * 32;
    __shared__ float s_acc[W > 1 ? 8 : 1][2][W > 1 ? D : 1];
    __shared__ float s_ml[8][2][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = warp % W;
    const int row_global = blockIdx.x * (8 / W) + warp / W;
    const int group = row_global / p.rows_per_slot;
    const int row = row_global - group * p.rows_per_slot;
    bool live = group < p.n_groups;
    DevMerge g{};
    DevReq rq{};
    if (live) { g = p.groups[group]; rq = p.reqs[g.req]; }
    const int tok = g.row_block * p.tokens_per_block + row / p.G;     // query row inside the request
    live = live && tok < rq.q_len;
    pdl_wait();
    pdl_trigger();

    float M[2] = {-INFINITY, -INFINITY}, L[2] = {0.f, 0.f}, acc[2][VEC];      // context, other
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[0][v] = acc[1][v] = 0.f;
    if (live) {
        #pragma unroll
        for (int seg = 0; seg < 2; ++seg) {
            const float* ws_o = seg ? p.ws_o : p.ws_o_ctx;
            const float* ws_ml = seg ? p.ws_ml : p.ws_ml_ctx;
            const int n = seg ? g.oth_n : g.ctx_n, stride = seg ? g.slot_stride : g.ctx_stride;
            const int per_slot = seg ? p.rows_per_slot : p.rows_per_slot_ctx;
            const size_t row0 = static_cast<size_t>(seg ? g.oth_slot0 : g.ctx_slot0) * per_slot + row + (seg ? 0 : g.ctx_row_off);
            const size_t step = static_cast<size_t>(stride) * per_slot;        // rows between consecutive partials
            if (W > 1 && n <= W) {
                // at most a partial per warp: it is the warp's result as it is, without the shuffles of two segments (2 requests' decode step
                // over 20 x 256 tokens 13.2 us per call, 12.6 this way; on inputs that stay in L2 9.3 and 8.6)
                if (part < n) {
                    const float2 ml = *reinterpret_cast<const float2*>(ws_ml + (row0 + part * step) * 2);
                    const float* a = ws_o + (row0 + part * step) * D + lane * VEC;
                    float x[VEC];
                    if constexpr (VEC == 4) { const float4 t = *reinterpret_cast<const float4*>(a); x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w; }
                    else { const float2 t = *reinterpret_cast<const float2*>(a); x[0] = t.x; x[1] = t.y; }
                    if (ml.y > 0.f) {
                        M[seg] = ml.x; L[seg] = ml.y;
                        #pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[seg][v] = x[v];
                    }
                }
                continue;
            }
            #pragma unroll 1
            for (int i0 = part; i0 < n; i0 += 32 * W) {
                const int mine = i0 + lane * W;                                // this lane's partial
                float2 ml = make_float2(-INFINITY, 0.f);
                if (mine < n) ml = *reinterpret_cast<const float2*>(ws_ml + (row0 + mine * step) * 2);
                const int cnt = min(32, (n - i0 + W - 1) / W);
                const float* src = ws_o + (row0 + i0 * step) * D + lane * VEC;
                const size_t src_step = static_cast<size_t>(W) * step * D;
                auto load = [&](int j, float (&x)[VEC]) {
                    const float* a = src + j * src_step;
                    if constexpr (VEC == 4) { const float4 t = *reinterpret_cast<const float4*>(a); x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w; }
                    else { const float2 t = *reinterpret_cast<const float2*>(a); x[0] = t.x; x[1] = t.y; }
                };
                float x[kBatch][VEC];
                // Requested together with (m, l): the row of an empty partial was never written, but it lies inside the
                // workspace, and the fold below never looks at what was read from it.
                #pragma unroll
                for (int u = 0; u < kBatch; ++u) if (u < cnt) load(u, x[u]);
                if (!(ml.y > 0.f)) ml = make_float2(-INFINITY, 0.f);           // empty partial
                float top = fmaxf(M[seg], ml.x);
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
                const float base = (top == -INFINITY) ? 0.f : top;
                const float f = (ml.y > 0.f) ? fast_exp2(ml.x - base) : 0.f, f_old = fast_exp2(M[seg] - base);
                float sum = ml.y * f;
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                L[seg] = L[seg] * f_old + sum;
                M[seg] = top;
                #pragma unroll
                for (int v = 0; v < VEC; ++v) acc[seg][v] *= f_old;
                #pragma unroll 1
                for (int j0 = 0; j0 < cnt; j0 += kBatch) {
                    if (j0 > 0) {
                        #pragma unroll
                        for (int u = 0; u < kBatch; ++u) if (j0 + u < cnt) load(j0 + u, x[u]);
                    }
                    #pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const float fj = __shfl_sync(0xffffffffu, f, (j0 + u) & 31);
                        if (j0 + u >= cnt || fj == 0.f) continue;
                        #pragma unroll
                        for (int v = 0; v < VEC; ++v) acc[seg][v] += x[u][v] * fj;
                    }
                }
            }
        }
    }
    if constexpr (W > 1) {
        #pragma unroll
        for (int seg = 0; seg < 2; ++seg) {
            #pragma unroll
            for (int v = 0; v < VEC; ++v) s_acc[warp][seg][lane * VEC + v] = acc[seg][v];
            if (lane == 0) { s_ml[warp][seg][0] = M[seg]; s_ml[warp][seg][1] = L[seg]; }
        }
        __syncthreads();
        if (part != 0) return;
        #pragma unroll
        for (int seg = 0; seg < 2; ++seg) {
            float top = -INFINITY;
            #pragma unroll
            for (int k = 0; k < W; ++k) top = fmaxf(top, s_ml[warp + k][seg][0]);
            const float base = (top == -INFINITY) ? 0.f : top;
            float sum = 0.f;
            #pragma unroll
            for (int v = 0; v < VEC; ++v) acc[seg][v] = 0.f;
            #pragma unroll
            for (int k = 0; k < W; ++k) {
                const float f = fast_exp2(s_ml[warp + k][seg][0] - base);
                sum += s_ml[warp + k][seg][1] * f;
                #pragma unroll
                for (int v = 0; v < VEC; ++v) acc[seg][v] += s_acc[warp + k][seg][lane * VEC + v] * f;
            }
            M[seg] = top; L[seg] = sum;
        }
    }
    if (!live) return;
    finish_row<VEC>(p, rq.q_row0 + tok, g.kv_head * p.G + row % p.G, lane, M, L, acc);
}

// Eq. 5 form for rows of few partials (at most kRowPartials a segment): eight lanes to a row, so that a warp has the loads of four rows
// under way, and every lane reads a row's (m, l) itself instead of twenty shuffles a row.  Bound by the latency of the loads.
constexpr int kRowPartials = 8;
template <int VEC>
__global__ void __launch_bounds__(128, 4) ape_merge_rows_kernel(const MergeParams p)
{
    constexpr int kBatch = 3;
    constexpr int D = VEC * 8;
    const int lane = threadIdx.x & 7;
    const int row_global = blockIdx.x * (blockDim.x / 8) + threadIdx.x / 8;
    const int group = row_global / p.rows_per_slot;
    const int row = row_global - group * p.rows_per_slot;
    bool live = group < p.n_groups;
    DevMerge g{};
    DevReq rq{};
    if (live) { g = p.groups[group]; rq = p.reqs[g.req]; }
    const int tok = g.row_block * p.tokens_per_block + row / p.G;     // query row inside the request
    live = live && tok < rq.q_len;
    pdl_wait();
    pdl_trigger();
    if (!live) return;
    float M[2], L[2], acc[2][VEC];                                    // context, other
    #pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
        const int n = seg ? g.oth_n : g.ctx_n, per_slot = seg ? p.rows_per_slot : p.rows_per_slot_ctx;
        const size_t row0 = static_cast<size_t>(seg ? g.oth_slot0 : g.ctx_slot0) * per_slot + row + (seg ? 0 : g.ctx_row_off);
        const size_t step = static_cast<size_t>(seg ? g.slot_stride : g.ctx_stride) * per_slot;        // rows between consecutive partials
        const float2* ml_at = reinterpret_cast<const float2*>(seg ? p.ws_ml : p.ws_ml_ctx) + row0;
        const float* src = (seg ? p.ws_o : p.ws_o_ctx) + row0 * D + lane * 4;
        float2 ml[kRowPartials];
        #pragma unroll
        for (int j = 0; j < kRowPartials; ++j) ml[j] = (j < n) ? ml_at[j * step] : make_float2(-INFINITY, 0.f);
        float x[kBatch][VEC];
        // The row of an empty partial was never written, but it lies inside the workspace, and the fold never looks at what was read from it.
        auto load = [&](int j0) {
            #pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (j0 + u < n) {
                    #pragma unroll
                    for (int v = 0; v < VEC; v += 4) {
                        const float4 t = *reinterpret_cast<const float4*>(src + (j0 + u) * step * D + v * 8);
                        x[u][v] = t.x; x[u][v + 1] = t.y; x[u][v + 2] = t.z; x[u][v + 3] = t.w;
                    }
                }
        };
        load(0);
        float top = -INFINITY, sum = 0.f;
        #pragma unroll
        for (int j = 0; j < kRowPartials; ++j) top = fmaxf(top, (ml[j].y > 0.f) ? ml[j].x : -INFINITY);       // (empty partial: no positive sum)
        const float base = (top == -INFINITY) ? 0.f : top;
        #pragma unroll
        for (int v = 0; v < VEC; ++v) acc[seg][v] = 0.f;
        #pragma unroll
        for (int j0 = 0; j0 < kRowPartials; j0 += kBatch) {
            if (j0 >= n) break;
            if (j0 > 0) load(j0);
            #pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (j0 + u < kRowPartials && j0 + u < n && ml[j0 + u].y > 0.f) {
                    const float f = fast_exp2(ml[j0 + u].x - base);
                    sum += ml[j0 + u].y * f;
                    #pragma unroll
                    for (int v = 0; v < VEC; ++v) acc[seg][v] += x[u][v] * f;
                }
        }
        M[seg] = top; L[seg] = sum;
    }
    finish_row<VEC, 8>(p, rq.q_row0 + tok, g.kv_head * p.G + row % p.G, lane, M, L, acc);
}

// Plans of the per-context form and of context trees that keep a partial per node (decode; prefill of few nodes): one warp per output row
// walks the partials in order.
template <int VEC, bool TREE>
__global__ void __launch_bounds__(256, 2) ape_merge_nodes_kernel(const MergeParams p)
{
    const int warp_global = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int group = warp_global / p.rows_per_slot;
    const int row = warp_global - group * p.rows_per_slot;
    pdl_wait();
    pdl_trigger();
    if (group >= p.n_groups) return;
    const DevMerge g = p.groups[group];
    const DevReq rq = p.reqs[g.req];
    const int tok = g.row_block * p.tokens_per_block + row / p.G;     // query row inside the request
    if (tok >= rq.q_len) return;

    float lse_c, norm_c, ac[VEC], Mo, Lo, ao[VEC];
    if constexpr (TREE) combine_tree<VEC>(p, g, row, lane, lse_c, norm_c, ac);
    else combine_per_context<VEC>(p, g, row, lane, lse_c, norm_c, ac);
    combine_segment<VEC>(p.ws_o, p.ws_ml, g.oth_slot0, g.oth_n, g.slot_stride, p.rows_per_slot, row, p.D, lane, Mo, Lo, ao);
    const float lse_o = (Lo > 0.f) ? (Mo + fast_log2(Lo)) : -INFINITY;
    write_row<VEC>(p, rq.q_row0 + tok, g.kv_head * p.G + row % p.G, lane, lse_c, norm_c, ac, lse_o, Lo, ao);
}

// Shards of a context-sharded attend (each holds a subset of the contexts): LSE_C = log sum_s e^{LSE_s},
// O_C = sum_s e^{LSE_s - LSE_C} O_s (appendix "Hierarchical Formula for Softmax Attention"), then Eq. 5 as above.
template <int VEC>
__global__ void __launch_bounds__(256) ape_shard_merge_kernel(const ShardMergeParams p)
{
    constexpr float kLog2e = 1.4426950408889634f;
    const int64_t warp_global = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp_global >= p.n_rows * p.H_q) return;
    const int64_t row = warp_global / p.H_q;
    const int h = static_cast<int>(warp_global - row * p.H_q);
    float M = -INFINITY, Z = 0.f, acc[VEC];
    #pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    for (int s = 0; s < p.n_shards; ++s) {
        const int64_t rh = (static_cast<int64_t>(s) * p.n_rows + row) * p.H_q + h;
        const float l = p.lse_ctx[rh] * kLog2e;
        if (!(l > -INFINITY)) continue;
        const float Mn = fmaxf(M, l);
        const float f_old = fast_exp2(M - Mn), f_new = fast_exp2(l - Mn);
        #pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] = acc[v] * f_old + p.o_ctx[rh * p.D + lane * VEC + v] * f_new;
        Z = Z * f_old + f_new;
        M = Mn;
    }
    const float lse_c = (Z > 0.f) ? p.S * (M + fast_log2(Z)) : -INFINITY;
    const int64_t rh = row * p.H_q + h;
    const float lo_nat = p.lse_oth[rh];
    const float lse_o = (lo_nat > -INFINITY) ? lo_nat * kLog2e : -INFINITY;
    const float top = fmaxf(lse_c, lse_o);
    float wc = 0.f, wo = 0.f, lam = -INFINITY;
    if (top > -INFINITY) {
        const float ec = fast_exp2(lse_c - top), eo = fast_exp2(lse_o - top);
        const float inv = 1.f / (ec + eo);
        wc = (Z > 0.f) ? ec * inv / Z : 0.f;
        wo = (lse_o > -INFINITY) ? eo * inv : 0.f;
        lam = (top + fast_log2(ec + eo)) * kLn2;
    }
    __nv_bfloat16* dst = p.out.data + row * p.out.token_stride + static_cast<int64_t>(h) * p.out.head_stride + lane * VEC;
    float r[VEC];
    #pragma unroll
    for (int v = 0; v < VEC; ++v) r[v] = wc * acc[v] + wo * p.o_oth[rh * p.D + lane * VEC + v];
    if constexpr (VEC == 4) {
        uint2 pk; pk.x = pack_bf16x2(r[0], r[1]); pk.y = pack_bf16x2(r[2], r[3]);
        *reinterpret_cast<uint2*>(dst) = pk;
    } else {
        *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(r[0], r[1]);
    }
    if (p.lse_out != nullptr && lane == 0) p.lse_out[rh] = lam;
}

}  // namespace

cudaError_t launch_shard_merge(const ShardMergeParams& p, cudaStream_t stream)
{
    const long long warps = static_cast<long long>(p.n_rows) * p.H_q;
    if (warps == 0) return cudaSuccess;
    const int blocks = static_cast<int>((warps * 32 + 255) / 256);
    return launch_kernel(false, p.D == 128 ? ape_shard_merge_kernel<4> : ape_shard_merge_kernel<2>, blocks, 256, 0, stream, p);
}

namespace {

__device__ __forceinline__ float logaddexp2(float a, float b) {
    const float m = fmaxf(a, b);
    if (m == -INFINITY) return -INFINITY;
    return m + log2f(exp2f(a - m) + exp2f(b - m));
}

// One thread per query row (token, head) of a request; consecutive threads hold consecutive rows, so every access to the
// [node][row] arrays is coalesced.
__global__ void __launch_bounds__(256)
ape_node_bias_kernel(const NodeBiasParams p)
{
    const int r = blockIdx.y;
    const DevReq rq = p.reqs[r];
    pdl_wait();
    pdl_trigger();
    const int64_t local = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (local >= static_cast<int64_t>(rq.q_len) * p.H_q) return;
    const int64_t row = static_cast<int64_t>(rq.pad) * p.H_q + local;
    const int n0 = p.req_node0[r], n1 = p.req_node0[r + 1];
    for (int n = n0; n < n1; ++n) p.mass[static_cast<int64_t>(n) * p.stat_rows + row] = -INFINITY;
    for (int n = n1 - 1; n >= n0; --n) {                     // children before parents
        const DevNode nd = p.nodes[n];
        float own = -INFINITY;
        if (nd.pad) {
            const float2 st = p.stats[static_cast<int64_t>(n) * p.stat_rows + row];
            if (st.y > 0.f) own = st.x + log2f(st.y);
        }
        const float A = logaddexp2(own, p.mass[static_cast<int64_t>(n) * p.stat_rows + row]);
        p.mass[static_cast<int64_t>(n) * p.stat_rows + row] = A;
        if (nd.parent >= 0) {
            float* up = p.mass + static_cast<int64_t>(nd.parent) * p.stat_rows + row;
            *up = logaddexp2(*up, nd.scaled ? p.S * A : A);
        }
    }
    for (int n = n0; n < n1; ++n) {                          // parents before children
        const DevNode nd = p.nodes[n];
        const float A = p.mass[static_cast<int64_t>(n) * p.stat_rows + row];
        float b = (nd.parent >= 0) ? p.bias[static_cast<int64_t>(nd.parent) * p.stat_rows + row] : 0.f;
        if (nd.scaled && A > -INFINITY) b += (p.S - 1.f) * A;
        p.bias[static_cast<int64_t>(n) * p.stat_rows + row] = b;
    }
}

// The same computation with a request's nodes x 32 rows in shared memory: a CTA takes 32 consecutive rows (lane = row), its warps
// share the nodes of a level.  The nodes come in breadth-first order, so that a level is a range and a node's children are a
// range of the next level: bottom-up a node gathers its children, top-down it adds to its parent's bias, one block barrier per
// level.  Bound by the statistics it reads and the biases it writes (12 bytes per node and row); walked node by node by one
// warp, the 128K prefill with 500 contexts spent 73 us here, by levels 27 us.
constexpr int kBiasRows = 32;
constexpr int kBiasWarps = 16;
__global__ void __launch_bounds__(kBiasWarps * 32)
ape_node_bias_smem_kernel(const NodeBiasParams p)
{
    extern __shared__ float val[];                           // [nodes of the request][32]: own mass, then A_n, then the bias
    const int r = blockIdx.y;
    const DevReq rq = p.reqs[r];
    const int64_t n_rows = static_cast<int64_t>(rq.q_len) * p.H_q;
    const int64_t local = static_cast<int64_t>(blockIdx.x) * kBiasRows + (threadIdx.x & 31);
    if (static_cast<int64_t>(blockIdx.x) * kBiasRows >= n_rows) return;
    const bool live = local < n_rows;
    const int64_t row = static_cast<int64_t>(rq.pad) * p.H_q + (live ? local : 0);
    const int n0 = p.req_node0[r], n_nodes = p.req_node0[r + 1] - n0;
    const int32_t* level = p.levels + static_cast<int64_t>(r) * kLevelStride;      // number of levels, then their ranges
    const int n_levels = level[0];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the node records behind the values, so that the walks read shared memory only
    DevBfsNode* rec = reinterpret_cast<DevBfsNode*>(val + static_cast<size_t>(n_nodes) * kBiasRows);
    for (int i = threadIdx.x; i < n_nodes; i += kBiasWarps * 32) rec[i] = p.bfs[n0 + i];
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    #pragma unroll 8
    for (int i = warp; i < n_nodes; i += kBiasWarps) {       // independent loads: several in flight per warp
        float2 st = make_float2(0.f, 0.f);
        if (live && (rec[i].a & BFS_TOKENS)) st = p.stats[static_cast<int64_t>(n0 + (rec[i].a & BFS_MASK)) * p.stat_rows + row];
        val[i * kBiasRows + lane] = (st.y > 0.f) ? st.x + fast_log2(st.y) : -INFINITY;
    }
    for (int lv = n_levels - 2; lv >= 0; --lv) {             // children before parents
        __syncthreads();
        for (int i = level[1 + lv] + warp; i < level[2 + lv]; i += kBiasWarps) {
            const int c0 = rec[i].b & BFS_MASK, c1 = (rec[i].b >> 12) & BFS_MASK;
            if (c0 == c1) continue;
            const float own = val[i * kBiasRows + lane];
            float top = own;
            for (int c = c0; c < c1; ++c) {
                const float A = val[c * kBiasRows + lane];
                top = fmaxf(top, (rec[c].a & BFS_SCALED) ? p.S * A : A);
            }
            if (top == -INFINITY) continue;
            float sum = fast_exp2(own - top);
            for (int c = c0; c < c1; ++c) {
                const float A = val[c * kBiasRows + lane];
                sum += fast_exp2(((rec[c].a & BFS_SCALED) ? p.S * A : A) - top);
            }
            val[i * kBiasRows + lane] = top + fast_log2(sum);
        }
    }
    for (int lv = 0; lv < n_levels; ++lv) {                  // parents before children
        if (n_levels > 1) __syncthreads();                   // (with one level a thread only meets its own values)
        for (int i = level[1 + lv] + warp; i < level[2 + lv]; i += kBiasWarps) {
            const DevBfsNode nd = rec[i];
            const float A = val[i * kBiasRows + lane];
            const int up = static_cast<int>((nd.a >> 12) & BFS_MASK) - 1;
            float b = (up >= 0) ? val[up * kBiasRows + lane] : 0.f;
            if ((nd.a & BFS_SCALED) && A > -INFINITY) b += (p.S - 1.f) * A;
            val[i * kBiasRows + lane] = b;
            if (live) p.bias[static_cast<int64_t>(n0 + (nd.a & BFS_MASK)) * p.stat_rows + row] = b;
        }
    }
}

}  // namespace

cudaError_t launch_node_bias(const NodeBiasParams& p, cudaStream_t stream)
{
    if (p.n_req <= 0 || p.max_rows <= 0) return cudaSuccess;
    const size_t smem = static_cast<size_t>(p.max_nodes) * (kBiasRows * sizeof(float) + sizeof(DevBfsNode));
    if (p.max_nodes > 0 && smem <= p.smem_limit) {
        // (the device's limit, not this launch's size: another thread may be between its own two steps)
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(ape_node_bias_smem_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       static_cast<int>(p.smem_limit));
            if (e != cudaSuccess) return e;
        }
        const dim3 grid(static_cast<unsigned>((p.max_rows + kBiasRows - 1) / kBiasRows), static_cast<unsigned>(p.n_req));
        return launch_pdl(ape_node_bias_smem_kernel, grid, kBiasWarps * 32, smem, stream, p);
    }
    // too many nodes for shared memory: the per-node arrays stay in global memory
    const dim3 grid(static_cast<unsigned>((p.max_rows + 255) / 256), static_cast<unsigned>(p.n_req));
    return launch_pdl(ape_node_bias_kernel, grid, 256, 0, stream, p);
}

namespace {
template <int VEC>
cudaError_t launch_merge_vec(const MergeParams& p, long long rows, cudaStream_t stream) {
    if (p.per_context != 0)
        return launch_pdl(p.per_context == 2 ? ape_merge_nodes_kernel<VEC, true> : ape_merge_nodes_kernel<VEC, false>,
                          static_cast<unsigned>((rows + 7) / 8), 256, 0, stream, p);
    // Eight warps per row while all rows' blocks are resident at once (four to an SM): with few rows, as in a decode step,
    // it is the latency of a row's partials that counts (4 requests over 20K tokens each: 62.1 us per step with one warp per row,
    // 60.5 with eight; 16 requests over shared 128K tokens: 129.0 and 124.4).  With more rows the warps of other rows hide it,
    // and sharing a row only adds the meeting in shared memory (64 rows over 10 x 256 tokens, 2048 rows to merge: 19.4 us with
    // one, 24.4 with eight; 4 x 128 rows over 20K tokens: 212 and 254).
    // With more rows than fit on the device at once that way (four blocks of eight to an SM) and few partials a segment (most prefills: the
    // runs of a head span few blocks), eight lanes take a row.  64 rows over 30 x 256 tokens, 3 / 4 requests (6,144 / 8,192 rows to merge):
    // 43.2 / 53.5 us per call with a warp per row, 41.2 / 50.9 this way; 2 x 256 rows over 20 x 256 tokens 68.3 and 64.2; 4 x 128 rows over 20
    // documents 200.7 and 196.7.  Below the line, 2 requests (4,096 rows) 28.9 and 29.5, a tree's 3,072 rows 54.8 and 55.8.
    if (rows > 32ll * p.n_sm && p.max_partials <= kRowPartials)
        return launch_pdl(ape_merge_rows_kernel<VEC * 4>, static_cast<unsigned>((rows + 15) / 16), 128, 0, stream, p);
    if (rows <= 4ll * p.n_sm) return launch_pdl(ape_merge_kernel<VEC, 8>, static_cast<unsigned>(rows), 256, 0, stream, p);
    return launch_pdl(ape_merge_kernel<VEC, 1>, static_cast<unsigned>((rows + 7) / 8), 256, 0, stream, p);
}
}  // namespace

cudaError_t launch_merge(const MergeParams& p, cudaStream_t stream)
{
    const long long rows = static_cast<long long>(p.n_groups) * p.rows_per_slot;
    if (rows == 0) return cudaSuccess;
    return p.D == 128 ? launch_merge_vec<4>(p, rows, stream) : launch_merge_vec<2>(p, rows, stream);
}

template <int VEC>
static cudaError_t merge_load_vec() {
    cudaFuncAttributes attr;
    for (auto* kernel : {ape_merge_kernel<VEC, 8>, ape_merge_kernel<VEC, 1>, ape_merge_rows_kernel<VEC * 4>}) {
        const cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
cudaError_t merge_load(int D) { return D == 128 ? merge_load_vec<4>() : merge_load_vec<2>(); }

}  // namespace ape
