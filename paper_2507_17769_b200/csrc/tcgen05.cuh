// What the three prefill kernels share: wrappers over the tcgen05 and tensor-map PTX they use, the matrix descriptors
// and the tensor maps of Q and the pool.
#pragma once

#include <cuda.h>

#include <cstring>

#include "common.cuh"

namespace ps {

// (entries past the list's end are not read)
inline void fill_inline_items(const RunArgs& a, InlineItems& inl) {
    if (!a.inline_items) return;
    memcpy(inl.item, a.inline_items, a.w.n_prefill * sizeof(PrefillItem));
    memcpy(inl.start, a.inline_starts, (a.w.n_prefill_ctas + 1) * sizeof(int32_t));
}

// Q as a [T tokens][Hq heads][D] tensor; a box is one 64-element half of a q tile's 128 (token, head) rows.
ps_status encode_q_map(const RunArgs& a, CUtensorMap* map);
// The pool as rows of 2 KB blocks (16 tokens x 64 elements); a box is one row, gathered four at a time.
constexpr int kPoolBlock = kPage * 128;
ps_status encode_pool_map(const RunArgs& a, CUtensorMap* map);

__host__ __device__ constexpr float scale_log2(int d) { return d == 128 ? 0.12751743f : 0.18033688f; }  // log2(e) / sqrt(d)

#ifdef __CUDACC__

__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One leader lane of a converged warp (always the same one for the full mask).  Issuing the MMAs under this
// predicate, rather than under a test of the lane index, keeps the descriptor arithmetic warp-uniform.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}" : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]
__device__ __forceinline__ void tc_mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem desc]
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
          "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
          "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
// 3-input max and packed fp32 pairs (two lanes per 64-bit register)
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
        "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15])
        : "memory");
}
// One box of a 3-d tensor map into shared memory; completion is counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Four 2 KB blocks of the pool, one after the other into shared memory (box: one row of the pool seen as rows of 2 KB; rows
// outside the pool read as zero).  A bulk copy per block costs the issuing warp some 100 cycles each, because its operands
// are uniform registers and the lanes take turns; with 8 of them the producers could not keep up (1500 cycles a key tile).
__device__ __forceinline__ void gather4(uint32_t dst, const CUtensorMap* map, int r0, int r1, int r2, int r3, uint32_t bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;" ::"r"(dst), "l"(map), "r"(0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar),
        "l"(policy)
        : "memory");
}
__device__ __forceinline__ void store_tagged(uint32_t addr, float v, uint32_t tag) {
    asm volatile("st.volatile.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(__float_as_uint(v)), "r"(tag) : "memory");
}
__device__ __forceinline__ uint32_t load_tagged(uint32_t addr, float& v) {
    uint32_t bits, tag;
    asm volatile("ld.volatile.shared.v2.b32 {%0, %1}, [%2];" : "=r"(bits), "=r"(tag) : "r"(addr) : "memory");
    v = __uint_as_float(bits);
    return tag;
}
__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
// 32 weights exp2(scale * s - ref) of one row as bf16 pairs, added to the packed row sums: two scores per instruction
// (packed fp32 FMA and add).  `top`: largest score so far.
template <int D>
__device__ __forceinline__ void weights32(const uint32_t (&s)[32], float ref, uint64_t& ls0, uint64_t& ls1, float& top, uint32_t* packed) {
    const uint64_t sc2 = pack2(scale_log2(D), scale_log2(D)), nm2 = pack2(-ref, -ref);
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
        top = max3(top, __uint_as_float(s[c]), __uint_as_float(s[c + 1]));
        float e0, e1;
        unpack2(fma2(pack2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, nm2), e0, e1);
        e0 = fast_exp2(e0), e1 = fast_exp2(e1);
        if (c & 2) ls1 = add2(ls1, pack2(e0, e1));
        else ls0 = add2(ls0, pack2(e0, e1));
        packed[c >> 1] = pack_bf16(e0, e1);
    }
}
// The same for the 64 scores of a half tile of which this row sees the first `vis`, and some row of the warp the first `vis_any`:
// masked by select.  l is the sum of the bf16-rounded weights that PV multiplies, so that the output of a row with a handful of keys
// stays an exact convex mix of V rows; `rounding` is what that adds to their exact sum, of which the log-sum-exp is taken.
// (Rolled: this code runs once or twice an item, so its instructions come from far; written out for all 64 scores it took 4700
// cycles a tile.  In steps of 16 scores, with the rounding added up weight by weight, four fresh prompts of 1400 to 2000 tokens took
// 120 us; so 111.)
template <int D>
__device__ __forceinline__ void masked_weights64(uint32_t s_addr, uint32_t p_addr, int vis, int vis_any, float ref, float& l, float& rounding) {
    const uint64_t sc2 = pack2(scale_log2(D), scale_log2(D)), nm2 = pack2(-ref, -ref);
    float l0 = 0.f, l1 = 0.f;
    uint64_t exact = 0ull;
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
        uint32_t packed[16];
        if (vis_any <= 32 * q) {
#pragma unroll
            for (int c = 0; c < 16; ++c) packed[c] = 0u;
        } else {
            uint32_t s[32];
            tmem_ld32(s_addr + 32 * q, s);
            tmem_wait_ld();
            const int v = vis - 32 * q;
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
                s[c] = c < v ? s[c] : 0xff800000u;
                s[c + 1] = c + 1 < v ? s[c + 1] : 0xff800000u;
                float e0, e1;
                unpack2(fma2(pack2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, nm2), e0, e1);
                e0 = fast_exp2(e0), e1 = fast_exp2(e1);
                exact = add2(exact, pack2(e0, e1));
                packed[c >> 1] = pack_bf16(e0, e1);
                l0 += bf16_lo(packed[c >> 1]);
                l1 += bf16_hi(packed[c >> 1]);
            }
        }
        tmem_st16(p_addr + 16 * q, packed);
    }
    float x0, x1;
    unpack2(exact, x0, x1);
    l += l0 + l1;
    rounding += (l0 - x0) + (l1 - x1);
}
// the largest of the first `vis` of them
__device__ __forceinline__ float masked_max64(uint32_t s_addr, int vis, int vis_any) {
    float mx = -INFINITY;
#pragma unroll 1
    for (int q = 0; q < 2 && 32 * q < vis_any; ++q) {
        uint32_t s[32];
        tmem_ld32(s_addr + 32 * q, s);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 32; ++c) mx = 32 * q + c < vis ? fmaxf(mx, __uint_as_float(s[c])) : mx;
    }
    return mx;
}
// 32 bytes to a 16-byte aligned address, in one store where it is 32-byte aligned
__device__ __forceinline__ void store32(char* dst, const uint32_t* v, bool aligned32) {
    if (aligned32) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                     "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    } else {
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(v[4], v[5], v[6], v[7]);
    }
}
// Shared-memory matrix descriptor, 128-byte swizzle, 8-row atoms of 1024 bytes.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version for this architecture
    d |= (uint64_t)2 << 61;  // SWIZZLE_128B
    return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, M x N.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}

#endif  // __CUDACC__

}  // namespace ps
