// Combine split-KV partial results.  For one query, attention over a union of
// disjoint key sets is the mix of the per-set results weighted by each set's
// exponential mass: with M = max_s lse_s,
//     out = sum_s e^{lse_s - M} o_s / sum_s e^{lse_s - M},  lse = M + log sum_s e^{lse_s - M}.
// Segments are combined in a fixed order, so the result is deterministic.
// Used for prefill q tile pairs cut into segments: a separate launch spreads the rows over all SMs (letting
// the last-arriving prefill CTA combine them instead was measured slower: one SM pulls the partial rows
// too slowly).  Decode rows are combined inside the decode kernel.
// A warp combines R output rows.  Their partial rows are requested before the log-sum-exps have arrived (their addresses
// do not depend on them), the log-sum-exps of all (row, segment) pairs are fetched one per lane, and the weights travel by
// shuffle, so the rows cost about one round trip to L2 together, after the entry record, which belongs to the run's own list and
// is read while the kernels before are still running.  (The partial rows are not read-only memory for this kernel: it may be there
// while the prefill kernel still writes them.  They are ordinary loads, behind the wait.)  Bound by latency: rows of few segments go four to a warp, so that all
// are under way at once (48 rows and two chunks at head dimension 64, whole iteration, 56.2 -> 55.3 us); rows of more than
// four segments, of which a batch has few, one to a warp with four segments in flight (100 tokens on 4000, ten segments, four rows
// a warp with two in flight: 18.5 -> 20.8).
#include <type_traits>

#include "common.cuh"

namespace ps {

namespace {

constexpr int kMergeWarps = 8;
constexpr int kFewSegs = 4;

// AHEAD: segments whose partial rows are in flight
template <int D, int R, int AHEAD>
__global__ void __launch_bounds__(kMergeWarps * 32) merge_kernel(const MergeEntry* __restrict__ entries,
                                                                  float* part_lse, float* part_o,
                                                                  __nv_bfloat16* __restrict__ out, float* __restrict__ lse,
                                                                  int Hq, int G) {
    constexpr int V = D / 32;  // floats per lane
    constexpr int kLaneSegs = 32 / R;  // segments of a row whose log-sum-exps the warp holds one per lane
    using Vec = typename std::conditional<V == 4, float4, float2>::type;
    const MergeEntry e = entries[blockIdx.x];
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = e.n_tok * G;
    const int rw0 = (warp + kMergeWarps * blockIdx.y) * R;
    if (rw0 >= rows) return;
    const int n_seg = e.n_seg;
    auto row_of = [&](int k) { return min(rw0 + k, rows - 1); };  // (past the end: a repeat that is not stored)
    auto row_ptr = [&](int k, int s) { return reinterpret_cast<const Vec*>(part_o + ((int64_t)e.base + row_of(k) + (int64_t)s * e.seg_stride) * D) + lane; };

    Vec x[R][AHEAD];
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
        for (int a = 0; a < AHEAD; ++a)
            if (a < n_seg) x[k][a] = *row_ptr(k, a);
    // Lanes kLaneSegs k .. have row k's segments.  A segment that saw no visible key for a row carries lse = -inf and weight 0.
    const float* const my_lse = part_lse + e.base + row_of(lane / kLaneSegs);
    auto lse_of = [&](int s) { return my_lse[(int64_t)s * e.seg_stride]; };
    const int my_seg = lane % kLaneSegs;
    const float lse_mine = my_seg < n_seg ? lse_of(my_seg) : -INFINITY;
    float M = lse_mine;
    for (int s = my_seg + kLaneSegs; s < n_seg; s += kLaneSegs) M = fmaxf(M, lse_of(s));
#pragma unroll
    for (int o = kLaneSegs / 2; o >= 1; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float w_mine = __expf(lse_mine - M);  // exp(-inf) = 0
    float denom = w_mine;
    for (int s = my_seg + kLaneSegs; s < n_seg; s += kLaneSegs) denom += __expf(lse_of(s) - M);
#pragma unroll
    for (int o = kLaneSegs / 2; o >= 1; o >>= 1) denom += __shfl_xor_sync(0xffffffffu, denom, o);

    float acc[R][V];
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
        for (int v = 0; v < V; ++v) acc[k][v] = 0.f;
    // segments in a fixed order, AHEAD of them at a time
    for (int s0 = 0; s0 < n_seg; s0 += AHEAD) {
        if (s0 > 0) {
#pragma unroll
            for (int k = 0; k < R; ++k)
#pragma unroll
                for (int a = 0; a < AHEAD; ++a)
                    if (s0 + a < n_seg) x[k][a] = *row_ptr(k, s0 + a);
        }
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
            const int s = s0 + a;
            if (s < n_seg) {  // warp-uniform
                const float w_far = s < kLaneSegs ? 0.f : __expf(lse_of(s) - M);  // of this lane's row
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float w = __shfl_sync(0xffffffffu, s < kLaneSegs ? w_mine : w_far, k * kLaneSegs + s % kLaneSegs);
                    acc[k][0] += w * x[k][a].x;
                    acc[k][1] += w * x[k][a].y;
                    if constexpr (V == 4) acc[k][2] += w * x[k][a].z, acc[k][3] += w * x[k][a].w;
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const float den = __shfl_sync(0xffffffffu, denom, k * kLaneSegs), top = __shfl_sync(0xffffffffu, M, k * kLaneSegs);
        const int rw = rw0 + k;
        if (rw < rows) {
            const float inv = 1.f / den;
            const int64_t orow = (int64_t)(e.q_tok + rw / G) * Hq + e.kv_head * G + rw % G;
            __nv_bfloat16* op = out + orow * D + lane * V;
            uint32_t y[V / 2];
#pragma unroll
            for (int v = 0; v < V; v += 2) y[v / 2] = pack_bf16(acc[k][v] * inv, acc[k][v + 1] * inv);
            if constexpr (V == 4) *reinterpret_cast<uint2*>(op) = make_uint2(y[0], y[1]);
            else *reinterpret_cast<uint32_t*>(op) = y[0];
            if (lse && lane == 0) lse[orow] = top + __logf(den);
        }
    }
}

}  // namespace

ps_status launch_merge(const RunArgs& a) {
    if (a.w.n_merge == 0) return PS_OK;
    const int Hq = a.shape.n_q_heads, G = Hq / a.shape.n_kv_heads;
    // blockIdx.x = merge entry (a prefill item cut into segments, up to 256 rows); blockIdx.y = its rows
    auto launch = [&](auto* kernel, int rows_of_warp) {
        return launch_kernel(kernel, dim3(a.w.n_merge, kPrefillRowsPerItem / (kMergeWarps * rows_of_warp)), kMergeWarps * 32, 0, a.stream, 1, a.early, a.w.merge,
                             a.w.part_lse, a.w.part_o, a.out, a.lse, Hq, G);
    };
    if (a.w.merge_segs <= kFewSegs) return a.shape.head_dim == 128 ? launch(merge_kernel<128, 4, 2>, 4) : launch(merge_kernel<64, 4, 2>, 4);
    return a.shape.head_dim == 128 ? launch(merge_kernel<128, 1, 4>, 1) : launch(merge_kernel<64, 1, 4>, 1);
}

}  // namespace ps
