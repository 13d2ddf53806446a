// Prefill-chunk attention for head dimension 128: a pair of CTAs per item.
//
// A chunk's rows attend the prior context plus the chunk's own earlier tokens (paper sections 2.4 and 4.7); this part is
// a dense contraction (section 3.4).  A cluster of two CTAs works through a list of items; an item = 256 (token, head)
// rows -- the G heads that share a kv head x 256 / G consecutive tokens -- over one key range.  Rank r of the pair holds
// rows 128 r .. 128 r + 127.  QK^T and PV run as tcgen05.mma with cta_group::2 (M = 256, N = 128), issued by rank 0: each
// CTA keeps half of every K and V tile in its shared memory and the tensor cores of both read both halves, so a CTA pulls
// 32 KB per 128-key step from L2 for 128 rows.
//
//   warps 0-15 softmax: thread = half a row (64 of a tile's 128 keys); warps 0-7 take the even key tiles, 8-15 the odd ones
//   warp 16    K producer: K half tiles (gathered pool blocks) and Q
//   warp 17    V producer
//   warp 18    rank 0: issues the MMAs; rank 1: tells rank 0 that this CTA's K and V half tiles and Q have landed
//   warp 19    rank 0: waits for V on the MMA warp's behalf; rank 1: fetches the pair's items, well ahead of their use
//
// TMEM columns (of each CTA): scores of key tile n at 128 (n % 3), O at 384.  Weights overwrite their own scores (bf16,
// each half in the first 32 of its 64 columns), so one barrier per tile says both that P is there and that the buffer may
// be written behind the PV that reads it: QK^T of tile n + 3 is issued right behind PV of tile n, three tiles ahead of use.
//
// The softmax needs no row maximum.  Weights are exp2 of the scaled scores less a reference, the maximum of 32 of the row's
// scores in the item's first tile: fp32 sums and accumulators and bf16 weights keep their relative precision wherever the
// exponents are, and the reference's own weight keeps a sum from being small.  An item with a row whose sum exceeds 2^100
// (scores of some 69 above the sample's, in natural units) is run again, first for its rows' maxima and then relative to them:
// 640 us instead of 240 on 2048 x 8192 if every item has such a row.  Rows that see fewer than 64 keys are always taken
// relative to their maximum.
//
// What bounds it: a 128-key step of the pair takes 1310 cycles, of which the tensor core needs 1024 and the exp2 unit as many.
// What is left is issue time: the MMA warp needs about 1150 cycles a step (16 MMAs and their commits 700, three
// waits), and every instruction that is not in a hot loop costs its warp some 6 cycles, because four softmax warps per
// scheduler evict it.  Hence one barrier per tile for that warp (a feeder warp waits for V on its behalf), gathered tensor
// copies, short code at the item's end, and items begun by the group that is not writing output.
// Measured (B200, 32 q / 8 kv heads, N(0,1) data, chunk x prior; kernel alone on all SMs, mean of 50 back to back between CUDA
// events, SM clock 1965 MHz), against one CTA per item with two q tiles in turn, P in tensor memory, running row maximum
// (prefill.cu), on the same GPU:
//     1536 x 3885  123.7 -> 100.0 us (1171 TFLOP/s, 0.70 of the measured cuBLAS burst rate)    512 x 8192  79.2 -> 67.8
//     2048 x 2048  116.5 -> 97.7    2048 x 8192  280.6 -> 222 us (1392 TFLOP/s, 0.83)
//     2 x 2048 on 19.8 k and 28.9 k, 64 q heads  3080 -> 2470 us (1380); in a long run power holds it to 2770 (1230, 0.87 of
//     cuBLAS's sustained rate).  Without the references and the rounding of the sums it takes 2 % less.
// Steps on the way, on 2048 x 8192 (shorter runs): pair with two score buffers and eight softmax warps 251 us; three buffers, sixteen
// warps, no maximum 245; warp-uniform MMA issue and the feeder 241; gathered copies 218; items begun by the other group and
// part of the exponentials as a polynomial on the FMA pipe 212.  (The polynomial was taken out again: beside the maximum that
// the sums' rounding needs it cost more than it saved, 278 us a run back to back with it and 263 without.)  Items fetched by a
// warp of their own: 888 items of one key tile (12 a pair) 70.5 -> 64 us, of five 112 -> 106, four prompts of 1400 to 2000
// tokens, whole iteration, 134.1 -> 129.5.
// Every wait is bounded; on expiry a CTA sets the timeout status and drains.
#include "tcgen05.cuh"

namespace ps {

namespace {

constexpr int kThreads = 640;
constexpr int kKProducerWarp = 16, kVProducerWarp = 17, kMmaWarp = 18, kItemWarp = 19;
constexpr int kRegsSoftmax = 104, kRegsOther = 64;  // 640 x 96 at launch = 512 x 104 + 128 x 64
constexpr int D = 128;
constexpr int kTileKeys = 128;
constexpr int kRows = 128;                // rows of one CTA
constexpr float kScaleLog2 = scale_log2(D);
// 2^-60, 2^100: row sums outside are recomputed.  (Below 2^100 the accumulators are finite for |V| up to 2^27; only a row whose
// sample was not finite can have a sum below 1.)
constexpr float kSumMin = 8.7e-19f, kSumMax = 1.26e30f;
constexpr int kStagesK = 4, kStagesV = 4;
static_assert(kStagesV <= 5, "the feeder counts on a key tile's weights being six tiles away from the next on its barrier");
constexpr int kScoreBufs = 3;
constexpr int kQBytes = 2 * kRows * 128;   // one CTA's Q tile: two 64-element halves
constexpr int kKBytes = 2 * 64 * 128;      // this CTA's 64 keys: two halves
constexpr int kVBytes = kTileKeys * 128;   // this CTA's 64 of the 128 output columns
constexpr int kOffQ = 0;
constexpr int kOffK = kOffQ + 2 * kQBytes;
constexpr int kOffV = kOffK + kStagesK * kKBytes;
constexpr int kOffBar = kOffV + kStagesV * kVBytes;
constexpr int kItemRing = 8;
// Key tiles of items fetched ahead.  An item's first K tile is used some 5000 cycles after its record is out, four key tiles;
// with 6 the tensor core waited for short items' K (four prompts of 1400 to 2000 tokens 131.4 us, with 12 129.5).
constexpr int kAheadTiles = 12;
// every warp of both CTAs but rank 1's item warp, which writes the records
constexpr int kRingConsumers = 2 * 20 - 1;
constexpr int64_t kPairDrainLimitNs = 100000000ll;
constexpr uint32_t kColO = 384;

struct Bars {  // byte offsets from the barrier block
    static constexpr int k_full = 0;                        // the half tile has landed (rank 0: and the peer's)
    static constexpr int k_empty = k_full + 8 * kStagesK;   // the MMAs that read the stage have retired
    static constexpr int v_full = k_empty + 8 * kStagesK;
    static constexpr int v_empty = v_full + 8 * kStagesV;
    static constexpr int q_full = v_empty + 8 * kStagesV, q_empty = q_full + 16;
    // Per tile mod 6, twice the buffers: a softmax warp skips the other group's tiles (up to three at an item's start) and the
    // feeder is up to four tiles ahead, and neither may take an older phase for the one it means.
    static constexpr int s_full = q_empty + 16;
    static constexpr int p_ready = s_full + 8 * 2 * kScoreBufs;  // rank 0: the softmax warps of both CTAs and the feeder
    static constexpr int o_done = p_ready + 8 * 2 * kScoreBufs;  // per item mod 4 (a warp that skips items then never skips a phase it could mistake)
    static constexpr int o_free = o_done + 32;              // rank 0
    static constexpr int mma_drained = o_free + 8;
    static constexpr int item_full = mma_drained + 8, item_empty = item_full + 8 * kItemRing;  // (item_empty: rank 1)
    static constexpr int n_bars = (item_empty + 8 * kItemRing) / 8;
    static constexpr int tmem_slot = item_empty + 8 * kItemRing, abort_slot = tmem_slot + 4, limit_slot = abort_slot + 4;
    static constexpr int armed = limit_slot + 4;            // parity of the last phase armed with copies: K, V stages, Q buffers
    static constexpr int n_armed = kStagesK + kStagesV + 2;
    static constexpr int again = armed + 4 * n_armed;       // rank 1, per ring slot a byte per rank and quarter of its rows: sums out of range
    static constexpr int ring = (again + 8 * kItemRing + 15) / 16 * 16;
    static constexpr int redo = ring + kItemRing * (int)sizeof(PrefillItem);      // rank 1: records to run again
    static constexpr int row_part = redo + kItemRing * (int)sizeof(PrefillItem);  // [item & 3][softmax warpgroup] per row: (sum or maximum, item number in the low byte of the sum's rounding)
    static constexpr int row_ref = row_part + 16 * kRows * 8;  // [item & 3] per row: (reference, item number)
    static constexpr int bytes = row_ref + 4 * kRows * 8;
};
constexpr int kSmemBytes = kOffBar + Bars::bytes + 1024;  // + alignment slack
static_assert(kSmemBytes <= 232448 && Bars::armed % 4 == 0 && sizeof(PrefillItem) == 32, "shared memory");
static_assert(kPrefillRowsPerItem == 2 * kRows, "an item is the rows of a CTA pair");
// In the ring a record's n_tok also says how the item is run (bits 24 up): as is, for its rows' maxima only, or relative to
// the maxima that the record before has found; in the last case bits 16 .. 23 are the quarters of either rank's rows to write.
constexpr uint32_t kModePlain = 0, kModeMax = 1, kModeRelative = 2;

struct PairParams {
    const char* pool;
    const int32_t* block_table;
    __nv_bfloat16* out;
    float* lse;
    WsHeader* hdr;
    const PrefillItem* items;
    const int32_t* pair_start;  // static partition: pair b runs items [pair_start[b], pair_start[b + 1]); null = dynamic queue
    float* part_lse;
    float* part_o;
    int64_t num_pages;
    uint32_t wait_limit_ns;
    int32_t max_pages;
    int32_t n_items;
    int32_t Hq, Hkv, G;
    int32_t n_req, total_q, n_part_slots;  // extents the item records are checked against
    int32_t tag;
    int32_t flags;
};
constexpr int32_t kOutAligned32 = 1, kInlineList = 2, kBeside = 4;
static_assert(sizeof(PairParams) <= 128, "parameter block");

// ---- cluster-wide variants of the wrappers ----------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void arrive_at(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void arrive_at_release_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// the same from one lane of a converged warp, without a branch
__device__ __forceinline__ void arrive_at_if(uint32_t cluster_bar, bool yes) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cluster.b64 _, [%0];\n\t}" ::"r"(cluster_bar),
                 "r"((uint32_t)yes)
                 : "memory");
}
__device__ __forceinline__ void store_at(uint32_t cluster_addr, uint4 v) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
// orders this thread's reads behind the completed phase at cluster scope (a fence would also wait for its output stores)
__device__ __forceinline__ void acquire_cluster(uint32_t bar, uint32_t parity) {
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%0], %1;\n\t}" ::"r"(bar), "r"(parity)
                 : "memory");
}
__device__ __forceinline__ void fence_cluster() { asm volatile("fence.acq_rel.cluster;" ::: "memory"); }
__device__ __forceinline__ void store_u8_at(uint32_t cluster_addr) {
    asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(cluster_addr), "h"((unsigned short)1) : "memory");
}
__device__ __forceinline__ void pair_tmem_alloc(uint32_t smem_dst, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void pair_tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void pair_tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void pair_mma_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void pair_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// arrives on the barrier at this offset in both CTAs once this thread's earlier MMAs have retired
__device__ __forceinline__ void pair_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((unsigned short)3)
        : "memory");
}

__global__ void __launch_bounds__(kThreads, 1) prefill_pair_kernel(const PairParams p, const __grid_constant__ CUtensorMap q_map,
                                                                    const __grid_constant__ CUtensorMap pool_map, const __grid_constant__ InlineItems inl) {
    extern __shared__ char smem_raw[];
    char* smem = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + kOffBar;
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kOffBar + Bars::abort_slot);
    // written by the producers' lane 0: parity of the last phase of each stage and buffer that was armed with copies
    // (-1: none yet); read only after an abort
    volatile int* const s_armed = reinterpret_cast<volatile int*>(smem + kOffBar + Bars::armed);
    // (through a shuffle, so that the compiler knows it to be warp-uniform and keeps the roles' counters, barrier addresses
    // and matrix descriptors in uniform registers)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 0) {
        s_abort[0] = 0;
        s_abort[1] = (int)p.wait_limit_ns;
    }
    if (warp == 0) {
        pair_tmem_alloc(bars + Bars::tmem_slot, 512);
        pair_tmem_relinquish();
    }
    const int tile_tok = kRows / p.G;
    const int g_shift = 31 - __clz(p.G);  // G is a power of two
    volatile uint8_t* const again = reinterpret_cast<volatile uint8_t*>(smem + kOffBar + Bars::again);
    uint4* const ring = reinterpret_cast<uint4*>(smem + kOffBar + Bars::ring);  // two uint4 per record
    uint4* const redo = reinterpret_cast<uint4*>(smem + kOffBar + Bars::redo);
    // next item of this pair's static share, or of the queue all pairs of the run drain
    const bool inline_list = (p.flags & kInlineList) != 0, static_share = inline_list || p.pair_start != nullptr;
    auto next_item = [&](int cur, int end) { return static_share ? (cur < end ? cur : p.n_items) : atomicAdd(&p.hdr->prefill_next, 1); };
    auto start_of = [&](int pair) { return inline_list ? inl.start[pair] : __ldg(p.pair_start + pair); };
    auto record = [&](int idx, uint4& a, uint4& b) {
        if (inline_list) {
            const PrefillItem& it = inl.item[idx];
            a = make_uint4(it.req, it.kv_head, it.key_begin, it.key_end);
            b = make_uint4(it.q_tok, it.n_tok, it.part_slot, it.first_pos);
        } else {
            a = __ldg(reinterpret_cast<const uint4*>(p.items + idx));
            b = __ldg(reinterpret_cast<const uint4*>(p.items + idx) + 1);
        }
    };
    if (rank == 1 && threadIdx.x == kItemWarp * 32) {
        // the first item's record is on its way before the pair meets
        const int pair = blockIdx.x >> 1;
        const int idx = next_item(static_share ? start_of(pair) : 0, static_share ? start_of(pair + 1) : 0);
        uint4 a = make_uint4(0, 0, 0, 0), b = a;
        if (idx < p.n_items) record(idx, a, b);
        redo[0] = a;
        redo[1] = b;
    }
    for (int k = threadIdx.x; k < Bars::n_bars; k += kThreads) {
        const int off = 8 * k;
        uint32_t count = 1;
        // rank 0: its own copies and the peer's relay
        if (off < Bars::k_empty || (off >= Bars::v_full && off < Bars::v_empty) || (off >= Bars::q_full && off < Bars::q_empty)) count = rank == 0 ? 2 : 1;
        else if (off >= Bars::p_ready && off < Bars::o_done) count = 17;
        else if (off == Bars::o_free) count = 16;
        else if (off >= Bars::item_empty) count = kRingConsumers;
        mbar_init(bars + off, count);
        mbar_fence_init();
    }
    for (int k = threadIdx.x; k < 20 * kRows; k += kThreads) store_tagged(bars + Bars::row_part + 8 * k, 0.f, 0xffffffffu);
    if (threadIdx.x < 8 * kItemRing) again[threadIdx.x] = 0;
    if (threadIdx.x < Bars::n_armed) s_armed[threadIdx.x] = -1;
    tc_fence_before();
    __syncthreads();
    if (!(p.flags & kBeside)) pdl_wait();
    cluster_sync();  // the peer's barriers are initialised before anything arrives at them
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(smem + kOffBar + Bars::tmem_slot), 0);
    const uint32_t lead = map_to_rank(bars, 0);   // rank 0's barrier block
    const uint32_t items = map_to_rank(bars, 1);  // rank 1's, where records are given back
    // warp-uniform result, so that the warp-collective instructions that follow stay converged
    auto wait_all = [](uint32_t bar, uint32_t parity, volatile int* abort_flag) {
        return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag));
    };
    constexpr uint32_t kIdescQK = instr_desc(2 * kRows, kTileKeys, false);
    constexpr uint32_t kIdescPV = instr_desc(2 * kRows, D, true);
    // consumer side of the record ring: record number n; false at the end-of-work record or on abort.  A softmax warp gives
    // the slot back when its part of the item's sums has been checked, so that a free slot means a checked item.
    auto take_record = [&](uint32_t n, uint4& a, uint4& b, bool give_back) -> bool {
        const uint32_t slot = n % kItemRing;
        if (!wait_all(bars + Bars::item_full + 8 * slot, (n / kItemRing) & 1, s_abort)) return false;
        acquire_cluster(bars + Bars::item_full + 8 * slot, (n / kItemRing) & 1);  // the record was written by rank 1
        a = ring[2 * slot];
        b = ring[2 * slot + 1];
        __syncwarp();
        if (give_back && lane == 0) arrive_at(items + Bars::item_empty + 8 * slot);
        return (int32_t)b.y > 0;
    };
    auto tiles_of = [](const uint4& a) { return ((int32_t)a.w - (int32_t)a.z + kTileKeys - 1) / kTileKeys; };

    if (warp < 16) {
        // ====================================================================
        // softmax: warpgroup 2 w + h takes keys 64 h .. 64 h + 63 of the key tiles of group w; thread t owns row t.  The
        // group that does not write the previous item's output begins an item with its first three tiles (as many as there
        // are score buffers), then the groups alternate.
        // ====================================================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        const uint32_t w = warp >> 3, h = (warp >> 2) & 1;
        const int t = threadIdx.x & 127;
        const uint32_t lane_tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        // this row's entry in slot [item & 3][warpgroup]
        auto row_part = [&](uint32_t item, uint32_t wg) { return bars + Bars::row_part + 8 * (((item & 3) * 4 + wg) * kRows + t); };
        auto row_ref = [&](uint32_t item) { return bars + Bars::row_ref + 8 * ((item & 3) * kRows + t); };
        // another warpgroup's entry for this row, once it carries `tag`
        auto read_tagged = [&](uint32_t addr, uint32_t item, float& v, float& rounding) -> bool {
            uint32_t t0 = 0;
            for (uint32_t i = 1;; ++i) {
                const uint32_t tag = load_tagged(addr, v);
                rounding = __uint_as_float(tag & ~0xffu);
                if (__all_sync(0xffffffffu, (tag & 0xffu) == (item & 0xffu))) return true;
                if ((i & (kWaitPollsPerClockRead - 1)) == 0 || s_abort[1] == 0) {
                    const uint32_t now = global_timer_lo() | 1u;
                    if (t0 == 0) t0 = now;
                    const bool out = *s_abort || now - t0 > (uint32_t)s_abort[1] || s_abort[1] == 0;
                    if (__any_sync(0xffffffffu, out)) {
                        *s_abort = 1;
                        return false;
                    }
                }
            }
        };
        uint32_t n_item = 0, tc0 = 0;  // tc0: number of the item's first key tile
        uint32_t g0 = 0;               // the group that begins the item
        bool ok = true;
        while (ok) {
            uint4 ra, rb;
            if (!take_record(n_item, ra, rb, false)) break;
            const int key_begin = (int)ra.z, key_end = (int)ra.w, n_tok = (int)(rb.y & 0xffffu), first_pos = (int)rb.w;
            const uint32_t mode = rb.y >> 24;
            const int n_tiles = tiles_of(ra);
            const int i = (int)rank * tile_tok + (t >> g_shift);  // token of this row within the item
            const int limit = min(first_pos + i + 1, key_end);     // first key this row does not see
            const int plain_keys = min(first_pos + (int)rank * tile_tok + 1, key_end);  // keys that every row of this CTA sees
            float rounding = 0.f;      // what rounding the weights has added to l
            float ref = 0.f, l = 0.f;  // l: sum of this thread's weights (or their maximum)
            float top = -INFINITY;     // largest score of its halves that needed no mask
            if (mode == kModeRelative) {
                ref = -INFINITY;
                for (uint32_t wg = 0; wg < 4 && ok; ++wg) {
                    float m, unused;
                    ok = read_tagged(row_part(n_item - 1, wg), n_item - 1, m, unused);
                    ref = fmaxf(ref, m);
                }
                if (!ok) break;
                if (ref == -INFINITY) ref = 0.f;
            }
            if (mode == kModeMax) l = -INFINITY;
            if (mode == kModePlain && w == g0) {
                // The row's reference, the same in both halves.  (Columns 32 to 63 hold scores until the tile's PV: a half's
                // weights go over its first 32.)
                const uint32_t buf6 = tc0 % (2 * kScoreBufs), buf = buf6 >= 3 ? buf6 - 3 : buf6;
                ok = wait_all(bars + Bars::s_full + 8 * buf6, (tc0 / (2 * kScoreBufs)) & 1, s_abort);
                if (!ok) break;
                tc_fence_after();
                uint32_t sv[32];
                tmem_ld32(lane_tm + buf * 128 + 32, sv);
                tmem_wait_ld();
                float mx = -INFINITY;
#pragma unroll
                for (int c = 0; c < 32; c += 2) mx = max3(mx, __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]));
                // (rows that see fewer than 64 keys: below; they are in items of at most three tiles)
                if (limit - key_begin >= 64 && fabsf(mx) < INFINITY) ref = mx * kScaleLog2;
                if (h == 0 && n_tiles > 3) store_tagged(row_ref(n_item), ref, n_item & 0xffu);
            } else if (mode == kModePlain && n_tiles > 3) {
                float unused;
                ok = read_tagged(row_ref(n_item), n_item, ref, unused);
                if (!ok) break;
            }
            for (int j = w == g0 ? 0 : 3; j < n_tiles; j += j < 2 ? 1 : 2) {
                const uint32_t tc = tc0 + j;
                const uint32_t buf6 = tc % (2 * kScoreBufs), buf = buf6 >= 3 ? buf6 - 3 : buf6;
                // (the first tile's scores have been waited for, for the reference)
                if (j > 0 || mode != kModePlain) ok = wait_all(bars + Bars::s_full + 8 * buf6, (tc / (2 * kScoreBufs)) & 1, s_abort);
                if (!ok) break;
                tc_fence_after();
                const uint32_t s_addr = lane_tm + buf * 128 + h * 64;
                const int tile_base = key_begin + j * kTileKeys;
                const int vis = limit - tile_base - (int)h * 64;  // columns [0, vis) of this half are visible to this row
                // columns of this half that every row of the warp sees (later rows see no fewer)
                const int vis_all = tile_base + kTileKeys <= plain_keys ? 64 : __shfl_sync(0xffffffffu, vis, 0);
                if (mode != kModeMax && vis_all >= 64) {
                    uint32_t s0[32], s1[32], packed[32];
                    tmem_ld32(s_addr, s0);
                    tmem_ld32(s_addr + 32, s1);
                    tmem_wait_ld();
                    uint64_t ls0 = 0ull, ls1 = 0ull;
                    weights32<D>(s0, ref, ls0, ls1, top, packed);
                    weights32<D>(s1, ref, ls0, ls1, top, packed + 16);
                    tmem_st32(s_addr, packed);
                    float a0, a1, a2, a3;
                    unpack2(ls0, a0, a1);
                    unpack2(ls1, a2, a3);
                    l += (a0 + a2) + (a1 + a3);
                } else {
                    // Diagonal and ragged halves, the only ones of rows with few visible keys.
                    const int vis_any = __shfl_sync(0xffffffffu, vis, 31);  // columns that some row of the warp sees
                    if (mode == kModePlain && j == 0 && h == 0 && __any_sync(0xffffffffu, vis < 64)) {
                        // Rows that see fewer than 64 keys of the item, all of them here: relative to their maximum, so that
                        // the weight that counts most is 1 and rounds to itself.  (Such rows do not average the weights'
                        // rounding out.  The item has at most three tiles then: this thread also writes their log-sum-exp.)
                        const float mx = masked_max64(s_addr, vis, vis_any);
                        if (vis < 64 && mx > -INFINITY) ref = mx * kScaleLog2;
                    }
                    if (mode == kModeMax) l = fmaxf(l, masked_max64(s_addr, vis, vis_any) * kScaleLog2);
                    else masked_weights64<D>(s_addr, s_addr, vis, vis_any, ref, l, rounding);
                }
                // keys at or past key_end: their V rows may be stale or poisoned; zero them so 0 * V = 0
                const int n_keys = key_end - tile_base;
                if (n_keys < kTileKeys && h == 0) {
                    const uint32_t s = tc % kStagesV;
                    ok = wait_all(bars + Bars::v_full + 8 * s, (tc / kStagesV) & 1, s_abort);
                    if (!ok) break;
                    if (t >= n_keys) {
                        char* vrow = smem + kOffV + s * kVBytes + t * 128;
#pragma unroll
                        for (int u = 0; u < 8; ++u) *reinterpret_cast<uint4*>(vrow + u * 16) = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                    fence_cluster();
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                arrive_at_if(lead + Bars::p_ready + 8 * buf6, lane == 0);
            }
            if (!ok) break;
            // ---- end of the item.  Every warpgroup leaves its sums; the two of the last tile wait for its PV and write the
            // output (64 columns each), the others go on with the next item, so that the tensor core does not run dry. ----
            const uint32_t g_last = n_tiles <= 3 ? g0 : g0 ^ (uint32_t)((n_tiles & 1) ^ 1);
            if (mode != kModeMax) {
                // PV multiplies rounded weights, and their sum is what normalises the output.  Where rounding matters a few keys
                // have most of the weight; counting it for the largest weight of each of a row's four threads leaves as small an
                // error as summing all the rounded weights (which would take two additions a pair of scores more).
                const float e = fast_exp2(fmaf(top, kScaleLog2, -ref)), d = bf16_lo(pack_bf16(e, 0.f)) - e;
                l += d;
                rounding += d;
            }
            store_tagged(row_part(n_item, 2 * w + h), l, (n_item & 0xffu) | (__float_as_uint(rounding) & ~0xffu));
            auto give_back = [&]() {
                __syncwarp();
                arrive_at_if(items + Bars::item_empty + 8 * (n_item % kItemRing), lane == 0);
            };
            if (g_last != w) {
                give_back();
            } else {
                // (the group that began the item first: which one that was depends on the items before)
                l = rounding = 0.f;
#pragma unroll 1
                for (uint32_t wg = 0; wg < 4 && ok; ++wg) {
                    float lp, rp;
                    ok = read_tagged(row_part(n_item, wg ^ (2 * g0)), n_item, lp, rp);
                    l += lp;
                    rounding += rp;
                }
                if (!ok) break;
                const float inv = l > 0.f ? 1.f / l : 0.f;
                const float lse_v = l > 0.f ? (ref + log2f(l - rounding)) * 0.6931471805599453f : -INFINITY;
                // (a row that sees no key of this item's range has an empty sum)
                const bool bad = i < n_tok && limit > key_begin && !(l >= kSumMin && l <= kSumMax);
                const uint32_t quarter = rank * 4 + (warp & 3);
                bool write = mode == kModeRelative ? ((rb.y >> (16 + quarter)) & 1u) != 0 : mode == kModePlain;
                if (mode == kModePlain && __any_sync(0xffffffffu, bad)) {
                    if (lane == 0) store_u8_at(items + Bars::again + 8 * (n_item % kItemRing) + quarter);
                    fence_cluster();
                    write = false;
                }
                give_back();
                const bool valid = i < n_tok && write;
                const int q_tok = (int)rb.x, part_slot = (int)rb.z, kv_head = (int)ra.y;
                const int64_t orow = (int64_t)(q_tok + i) * p.Hq + kv_head * p.G + (t & (p.G - 1));
                const int64_t prow = (int64_t)part_slot + (int64_t)rank * kRows + t;
                ok = wait_all(bars + Bars::o_done + 8 * (n_item & 3), (n_item >> 2) & 1, s_abort);
                if (!ok) break;
                tc_fence_after();
                uint32_t v[2][32];
                tmem_ld32(lane_tm + kColO + h * 64, v[0]);
                tmem_ld32(lane_tm + kColO + h * 64 + 32, v[1]);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                arrive_at_if(lead + Bars::o_free, lane == 0);
                // Every lane writes its own row, 32 bytes (a DRAM sector) at a time: staging the tile in shared memory for
                // wider contiguous stores took 2700 cycles of these warps' time.
                if (valid) {
                    if (part_slot < 0) {
                        char* dst = reinterpret_cast<char*>(p.out + orow * D + h * 64);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            uint32_t x[8];
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                x[c] = pack_bf16(__uint_as_float(v[u >> 1][(u & 1) * 16 + 2 * c]) * inv, __uint_as_float(v[u >> 1][(u & 1) * 16 + 2 * c + 1]) * inv);
                            store32(dst + 32 * u, x, p.flags & kOutAligned32);
                        }
                    } else {
                        char* dst = reinterpret_cast<char*>(p.part_o + prow * D + h * 64);
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            uint32_t x[8];
#pragma unroll
                            for (int c = 0; c < 8; ++c) x[c] = __float_as_uint(__uint_as_float(v[u >> 2][(u & 3) * 8 + c]) * inv);
                            store32(dst + 32 * u, x, true);
                        }
                    }
                }
                if (valid && h == 0) {
                    if (part_slot >= 0) p.part_lse[prow] = lse_v;
                    else if (p.lse) p.lse[orow] = lse_v;
                }
            }
            g0 = g_last ^ 1;
            tc0 += n_tiles;
            ++n_item;
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
        if (warp == kKProducerWarp || warp == kVProducerWarp) {
            // ================================================================
            // producers: K half tiles (this rank's 64 keys) with the Q tiles; V half tiles (this rank's 64 columns).  K/V tiles of a chunk's sequence are read again by every other item of that
            // sequence: they are marked last to leave L2.
            // ================================================================
            const bool is_k = warp == kKProducerWarp;
            const uint64_t kv_policy = l2_policy_evict_last();
            uint32_t n_item = 0, tc = 0;
            bool ok = true;
            for (; ok; ++n_item) {
                uint4 ra, rb;
                if (!take_record(n_item, ra, rb, true)) break;
                const int kv_head = (int)ra.y;
                const int key_begin = (int)ra.z;
                const int n_tiles = tiles_of(ra), n_pages = ((int)ra.w - key_begin + kPage - 1) / kPage;
                const int32_t* bt = p.block_table + (int64_t)(int32_t)ra.x * p.max_pages + key_begin / kPage;
                // Pool rows (2 KB blocks: K halves 0 and 1, V halves 0 and 1 of a page) of four tiles at a time, one page per
                // lane, requested four tiles ahead; -8 for a page that is not there.
                auto pool_row = [&](int page, int idx) {
                    const bool has = idx < n_pages, good = has && (uint32_t)page < (uint64_t)p.num_pages;
                    if (has && !good) report(p.hdr, p.tag, kStatusBounds);
                    return good ? (page * p.Hkv + kv_head) * 4 : -8;
                };
                int row = -8, bt_next = lane < n_pages ? __ldg(bt + lane) : 0;
                for (int j = 0; j < n_tiles; ++j, ++tc) {
                    if ((j & 3) == 0) {
                        row = pool_row(bt_next, j * 8 + lane);
                        bt_next = (j + 4) * 8 + lane < n_pages ? __ldg(bt + (j + 4) * 8 + lane) : 0;
                    }
                    // K: the four pages of this rank's keys; V: all eight, this rank's half of the columns
                    const int src = (j & 3) * 8 + (is_k ? (int)rank * 4 : 0);
                    int r[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) r[k] = __shfl_sync(0xffffffffu, row, (src + k) & 31) + (is_k ? 0 : 2 + (int)rank);
                    const uint32_t s = is_k ? tc % kStagesK : tc % kStagesV;
                    const uint32_t par = (is_k ? tc / kStagesK : tc / kStagesV) & 1;
                    const uint32_t land = bars + (is_k ? Bars::k_full : Bars::v_full) + 8 * s;
                    ok = wait_all(bars + (is_k ? Bars::k_empty : Bars::v_empty) + 8 * s, par ^ 1, s_abort);
                    if (!ok) break;
                    if (elect_one()) {
                        mbar_expect_tx(land, 8 * kPoolBlock);
                        s_armed[is_k ? s : kStagesK + s] = (int)par;
                        const uint32_t dst = sbase + (is_k ? kOffK + s * kKBytes : kOffV + s * kVBytes);
                        gather4(dst, &pool_map, r[0], r[1], r[2], r[3], land, kv_policy);
                        if (is_k) gather4(dst + 4 * kPoolBlock, &pool_map, r[0] + 1, r[1] + 1, r[2] + 1, r[3] + 1, land, kv_policy);
                        else gather4(dst + 4 * kPoolBlock, &pool_map, r[4], r[5], r[6], r[7], land, kv_policy);
                    }
                    __syncwarp();
                    if (is_k && j == 0) {
                        // this rank's Q tile: rows (token, head of the group) in token-major order, one box of
                        // [128 / G tokens][G heads][64 elements] per half, in the 128-byte swizzle
                        const uint32_t qb = n_item & 1, qpar = (n_item >> 1) & 1;
                        ok = wait_all(bars + Bars::q_empty + 8 * qb, qpar ^ 1, s_abort);
                        if (!ok) break;
                        if (lane == 0) {
                            mbar_expect_tx(bars + Bars::q_full + 8 * qb, kQBytes);
                            s_armed[kStagesK + kStagesV + qb] = (int)qpar;
#pragma unroll
                            for (int hf = 0; hf < 2; ++hf)
                                tma_load_3d(sbase + kOffQ + qb * kQBytes + hf * (kRows * 128), &q_map, hf * 64, kv_head * p.G,
                                            (int32_t)rb.x + (int)rank * tile_tok, bars + Bars::q_full + 8 * qb);
                        }
                        __syncwarp();
                    }
                }
            }
            // the arrivals that rank 0's commits still owe this CTA's barriers come before it leaves
            if (ok && !*s_abort) {
                const int n_st = is_k ? kStagesK : kStagesV;
                for (int s = 0; s < n_st && ok; ++s) {
                    const uint32_t uses = (tc + n_st - 1 - s) / n_st;  // key tiles that went through stage s
                    if (uses > 0) ok = wait_all(bars + (is_k ? Bars::k_empty : Bars::v_empty) + 8 * s, (uses - 1) & 1, s_abort);
                }
                for (uint32_t qb = 0; qb < 2 && is_k && ok; ++qb) {
                    const uint32_t uses = (n_item + 1 - qb) / 2;
                    if (uses > 0) ok = wait_all(bars + Bars::q_empty + 8 * qb, (uses - 1) & 1, s_abort);
                }
            }
        } else if (rank == 0 && warp == kMmaWarp) {
            // ================================================================
            // MMA issue: PV of key tile n as soon as its weights are there, and right behind it QK^T of tile n + 3 into the
            // same buffer (the tensor pipe runs this thread's MMAs in issue order)
            // ================================================================
            const uint64_t desc_k = smem_desc(0, 16, 1024);
            const uint64_t desc_v = smem_desc(0, kVBytes, 1024);
            uint32_t n_item = 0, ahead = 0;           // items begun; key tiles whose QK^T has been issued and whose PV has not
            uint32_t q_buf = 0, q_buf6 = 0, p_buf = 0, p_buf6 = 0, p_par = 0;  // tile number mod 3 and 6 of either stream
            uint32_t k_st = 0, k_par = 0, v_st = 0, qb = 1;
            uint32_t n_out = 0;                       // items whose last PV has been issued
            uint32_t lasts = 0, nq = 0, np = 0;       // bit n % 32: tile n is its item's last
            int left = 0;                             // key tiles of the item whose QK^T is still to come
            bool ok = true, more = true, first = true;
            const uint32_t q_lo = (sbase + kOffQ) >> 4, k_lo = (sbase + kOffK) >> 4, v_lo = (sbase + kOffV) >> 4;
            const uint32_t hi_k = (uint32_t)(desc_k >> 32), hi_v = (uint32_t)(desc_v >> 32);
            while (true) {
                if (more && ahead < kScoreBufs) {
                    if (left == 0) {
                        // (with PVs outstanding the next record is not waited for)
                        if (ahead > 0 && !__all_sync(0xffffffffu, mbar_test_wait(bars + Bars::item_full + 8 * (n_item % kItemRing), (n_item / kItemRing) & 1)))
                            goto issue_pv;
                        uint4 ra, rb;
                        more = take_record(n_item, ra, rb, true);
                        if (!more) continue;
                        left = __shfl_sync(0xffffffffu, tiles_of(ra), 0);
                        qb = n_item & 1;
                        ok = wait_all(bars + Bars::q_full + 8 * qb, (n_item >> 1) & 1, s_abort);
                        if (!ok) break;
                        ++n_item;
                    }
                    ok = wait_all(bars + Bars::k_full + 8 * k_st, k_par, s_abort);
                    if (!ok) break;
                    tc_fence_after();
                    --left;
                    if (elect_one()) {
                        const uint32_t d_addr = tmem + q_buf * 128;
                        const uint32_t q = (uint32_t)desc_k + q_lo + qb * (kQBytes >> 4), k = (uint32_t)desc_k + k_lo + k_st * (kKBytes >> 4);
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            pair_mma_ss(d_addr, desc64(q + (((kk >> 2) * (kRows * 128) + (kk & 3) * 32) >> 4), hi_k),
                                        desc64(k + (((kk >> 2) * (64 * 128) + (kk & 3) * 32) >> 4), hi_k), kIdescQK, kk > 0);
                        pair_commit(bars + Bars::s_full + 8 * q_buf6);
                        pair_commit(bars + Bars::k_empty + 8 * k_st);
                        if (left == 0) pair_commit(bars + Bars::q_empty + 8 * qb);
                    }
                    __syncwarp();
                    if (left == 0) lasts |= 1u << (nq & 31);
                    ++nq;
                    ++ahead;
                    q_buf = q_buf == 2 ? 0 : q_buf + 1;
                    q_buf6 = q_buf6 == 5 ? 0 : q_buf6 + 1;
                    k_st = (k_st + 1) % kStagesK;
                    k_par ^= k_st == 0 ? 1u : 0u;
                    if (ahead < kScoreBufs) continue;
                }
            issue_pv:
                if (ahead == 0) break;
                // the weights, and V, for which the feeder has waited
                ok = wait_all(bars + Bars::p_ready + 8 * p_buf6, p_par, s_abort);
                // (O is overwritten: the previous item's has been read)
                if (ok && first && n_out > 0) ok = wait_all(bars + Bars::o_free, (n_out - 1) & 1, s_abort);
                if (!ok) break;
                tc_fence_after();
                const bool last = (lasts >> (np & 31)) & 1u;
                if (elect_one()) {
                    const uint32_t v = (uint32_t)desc_v + v_lo + v_st * (kVBytes >> 4);
                    const uint32_t p_addr = tmem + p_buf * 128;
#pragma unroll
                    for (int kk = 0; kk < kTileKeys / 16; ++kk)
                        pair_mma_ts(tmem + kColO, p_addr + (kk >> 2) * 64 + (kk & 3) * 8, desc64(v + kk * (2048 >> 4), hi_v), kIdescPV,
                                    (!first || kk > 0) ? 1u : 0u);
                    pair_commit(bars + Bars::v_empty + 8 * v_st);
                    if (last) pair_commit(bars + Bars::o_done + 8 * (n_out & 3));
                }
                __syncwarp();
                first = last;
                if (last) {
                    lasts &= ~(1u << (np & 31));
                    ++n_out;
                }
                ++np;
                --ahead;
                p_buf = p_buf == 2 ? 0 : p_buf + 1;
                p_par ^= p_buf6 == 5 ? 1u : 0u;
                p_buf6 = p_buf6 == 5 ? 0 : p_buf6 + 1;
                v_st = (v_st + 1) % kStagesV;
            }
        } else if (rank == 0) {
            // ================================================================
            // feeder: does the MMA warp's waits for V and adds one arrival to the weights' barrier.  (A wait takes that warp
            // 140 cycles and more even when it need not wait; with three waits a tile the tensor core starved.)
            // ================================================================
            uint32_t n_item = 0, n = 0, buf6 = 0;
            bool ok = true;
            uint4 ra, rb;
            while (ok && take_record(n_item, ra, rb, true)) {
                const int n_tiles = tiles_of(ra);
                for (int j = 0; j < n_tiles; ++j, ++n) {
                    ok = wait_all(bars + Bars::v_full + 8 * (n % kStagesV), (n / kStagesV) & 1, s_abort);
                    if (!ok) break;
                    if (lane == 0) mbar_arrive(bars + Bars::p_ready + 8 * buf6);
                    buf6 = buf6 == 5 ? 0 : buf6 + 1;
                }
                ++n_item;
            }
        } else if (warp == kMmaWarp) {
            // ================================================================
            // relay: tells rank 0 that this CTA's half tiles have landed.  V follows K two tiles behind, which is about when
            // either is asked for, so that neither is told late; when no next record is out, V catches up first.  It also does
            // once the last record is out, which may be before the last two tiles' V has landed: the softmax warps give an
            // item back when its sums are checked, and only the one of a ragged last tile has waited for V.
            // ================================================================
            uint32_t n_item = 0, n = 0, nv = 0;  // key tiles whose K, and V, has been told of
            bool ok = true;
            uint4 ra, rb;
            auto tell_v = [&]() {
                const uint32_t s = nv % kStagesV;
                ok = wait_all(bars + Bars::v_full + 8 * s, (nv / kStagesV) & 1, s_abort);
                if (ok && lane == 0) arrive_at(lead + Bars::v_full + 8 * s);
                ++nv;
            };
            while (ok) {
                if (!__all_sync(0xffffffffu, mbar_test_wait(bars + Bars::item_full + 8 * (n_item % kItemRing), (n_item / kItemRing) & 1)))
                    while (ok && nv < n) tell_v();
                if (!ok || !take_record(n_item, ra, rb, true)) break;
                const int n_tiles = tiles_of(ra);
                for (int j = 0; j < n_tiles && ok; ++j) {
                    const uint32_t s = n % kStagesK;
                    ok = wait_all(bars + Bars::k_full + 8 * s, (n / kStagesK) & 1, s_abort);
                    if (!ok) break;
                    if (lane == 0) arrive_at(lead + Bars::k_full + 8 * s);
                    if (j == 0) {
                        ok = wait_all(bars + Bars::q_full + 8 * (n_item & 1), (n_item >> 1) & 1, s_abort);
                        if (!ok) break;
                        if (lane == 0) arrive_at(lead + Bars::q_full + 8 * (n_item & 1));
                    }
                    ++n;
                    while (ok && nv + 2 < n) tell_v();
                }
                ++n_item;
            }
            while (ok && nv < n) tell_v();
        } else {
            // ================================================================
            // items: fetches the pair's records, from its static share or the queue, and puts them into both CTAs' rings as
            // slots come free.  (Done by the K producer between its copies, an item cost 4.0 us beyond its key tiles: some 200
            // instructions that no hot loop keeps in the instruction cache, and two trips to L2.)
            // ================================================================
            const int pair = blockIdx.x >> 1;
            int static_cur = 0, static_end = 0;
            if (static_share) {
                static_cur = start_of(pair) + 1;
                static_end = start_of(pair + 1);
            }
            uint32_t mode = kModePlain, redo_head = 0, redo_tail = 0;  // records put aside
            uint4 fa = redo[0], fb = redo[1];                          // the record fetched; n_tok = 0: end of work
            uint4 na, nb;                                              // the record published last
            __syncwarp();  // (the ring of records put aside begins with the first one's place)
            auto check_record = [&]() {
                if ((int32_t)fb.y == 0) return;
                // A record that points outside the batch (only a damaged work list has one) ends this pair's work and
                // flags the run; nothing is read or written through it.
                const int32_t r_req = (int32_t)fa.x, r_g = (int32_t)fa.y, r_kb = (int32_t)fa.z, r_ke = (int32_t)fa.w;
                const int32_t r_q = (int32_t)fb.x, r_n = (int32_t)fb.y, r_slot = (int32_t)fb.z, r_pos = (int32_t)fb.w;
                const bool rec_ok = (uint32_t)r_req < (uint32_t)p.n_req && (uint32_t)r_g < (uint32_t)p.Hkv && r_kb >= 0 &&
                                    r_kb % kTileKeys == 0 && r_kb < r_ke && r_ke <= p.max_pages * kPage && r_n >= 1 &&
                                    r_n <= 2 * tile_tok && r_q >= 0 && (int64_t)r_q + r_n <= p.total_q && r_pos >= 0 &&
                                    (int64_t)r_pos + r_n >= r_ke &&
                                    (r_slot < 0 || (int64_t)r_slot + (int64_t)r_n * p.G <= p.n_part_slots);
                if (!rec_ok) {
                    if (lane == 0) report(p.hdr, p.tag, kStatusBounds);
                    fa = fb = make_uint4(0, 0, 0, 0);
                }
            };
            auto fetch_record = [&]() {
                int idx = 0;
                if (lane == 0) idx = next_item(static_cur, static_end);
                ++static_cur;
                idx = __shfl_sync(0xffffffffu, idx, 0);
                fa = fb = make_uint4(0, 0, 0, 0);
                if (idx < p.n_items) record(idx, fa, fb);
                check_record();
            };
            // every consumer is done with the record that last used the slot of record n; if its item has to be run again,
            // the record is put aside
            auto reclaim = [&](uint32_t n) -> bool {
                const uint32_t slot = n % kItemRing, par = ((n / kItemRing) & 1) ^ 1;
                if (!wait_all(bars + Bars::item_empty + 8 * slot, par, s_abort)) return false;
                acquire_cluster(bars + Bars::item_empty + 8 * slot, par);
                const uint32_t mask = __ballot_sync(0xffffffffu, lane < 8 && again[8 * slot + (lane & 7)] != 0);
                if (mask) {
                    if (lane < 2) {
                        uint4 x = ring[2 * slot + lane];
                        if (lane == 1) x.y |= mask << 16;
                        redo[2 * (redo_tail % kItemRing) + lane] = x;
                    }
                    ++redo_tail;
                    if (lane < 8) again[8 * slot + lane] = 0;
                    __syncwarp();
                }
                return true;
            };
            check_record();
            uint32_t done = 0;  // records known to be given back
            int out = 0;        // key tiles of the records published behind them
            // publishes record n: the second pass of an item run again, the first one of the next such item, or the record
            // fetched (which stays fetched in the first two cases)
            bool ok = true;
            for (uint32_t n = 0; ok; ++n) {
                if (!reclaim(n)) break;
                if (mode != kModeMax && redo_head == redo_tail && (int32_t)fb.y == 0) {
                    // end of work, unless one of the items still under way has to be run again
                    for (uint32_t k = 1; k < kItemRing && ok; ++k)
                        if (n >= k) ok = reclaim(n - k + kItemRing);
                    if (!ok) break;
                }
                bool from_fetched = false;
                if (mode == kModeMax) {
                    mode = kModeRelative;
                } else if (redo_head != redo_tail) {
                    na = redo[2 * (redo_head % kItemRing)];
                    nb = redo[2 * (redo_head % kItemRing) + 1];
                    ++redo_head;
                    mode = kModeMax;
                } else {
                    na = fa;
                    nb = fb;
                    mode = kModePlain;
                    from_fetched = true;
                }
                nb.y = (nb.y & 0xffffffu) | (mode << 24);
                const uint32_t slot = n % kItemRing;
                if (lane == 0) {
                    ring[2 * slot] = na;
                    ring[2 * slot + 1] = nb;
                    mbar_arrive(bars + Bars::item_full + 8 * slot);
                    store_at(lead + Bars::ring + 32 * slot, na);
                    store_at(lead + Bars::ring + 32 * slot + 16, nb);
                    arrive_at_release_cluster(lead + Bars::item_full + 8 * slot);
                }
                __syncwarp();
                if (from_fetched && (int32_t)nb.y == 0) break;
                // An item taken early from the queue is one that an idle pair cannot take: only one is, beyond kAheadTiles.  (And
                // `done` stays within a ring of n: a slot's barrier tells its last two phases apart, no more.)
                out += tiles_of(na);
                for (; ok && done < n && (out > kAheadTiles || n - done >= kItemRing - 1); ++done) {
                    ok = reclaim(done + kItemRing);
                    out -= tiles_of(ring[2 * (done % kItemRing)]);
                }
                if (ok && from_fetched) fetch_record();
            }
        }
    }

    // (not before: a kernel that waits for this one's end would take the place of the decode kernel's CTAs beside it)
    pdl_trigger();
    if (warp == kMmaWarp) {
        if (rank == 0) {
            if (elect_one()) pair_commit(bars + Bars::mma_drained);
            __syncwarp();
        }
        // (in both ranks: everything rank 0 has issued is done, so no arrival is on its way to this CTA any more)
        mbar_wait(bars + Bars::mma_drained, 0, kDrainLimitNs);
    }
    tc_fence_before();
    __syncthreads();  // every role of this CTA has left its loop
    if (*s_abort) {
        // A bounded wait ran out somewhere in this CTA: the output is invalid and the run is flagged.  Before the pair
        // gives back its shared and tensor memory, the copies requested get a bounded time to land (the MMAs have retired).
        if (threadIdx.x == 0) report(p.hdr, p.tag, kStatusTimeout);
        if (warp == kKProducerWarp) {
            // (rank 0's barriers also count the peer's relay, which may never come: the copies land in microseconds, so one
            // limit serves them all)
            const uint64_t t0 = global_timer_ns();
            for (int k = 0; k < Bars::n_armed; ++k) {
                const int par = s_armed[k];
                const int64_t left = kPairDrainLimitNs - (int64_t)(global_timer_ns() - t0);
                const int bar = k < kStagesK ? Bars::k_full + 8 * k
                                             : k < kStagesK + kStagesV ? Bars::v_full + 8 * (k - kStagesK)
                                                                       : Bars::q_full + 8 * (k - kStagesK - kStagesV);
                if (par >= 0) mbar_wait(bars + bar, (uint32_t)par, left);
            }
        }
        __syncthreads();
    }
    cluster_sync();
    if (warp == 0) pair_tmem_dealloc(tmem, 512);
    // This kernel's end also means that of the decode kernel beside it.  (One CTA's last instruction: what follows a wait is
    // time between this run and the next kernel.)
    if ((p.flags & kBeside) && blockIdx.x == 0) pdl_wait();
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up through the runtime so that the library does not link libcuda.
EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return (EncodeTiledFn)f;
    }();
    return fn;
}

}  // namespace

ps_status encode_q_map(const RunArgs& a, CUtensorMap* map) {
    EncodeTiledFn encode = tensor_map_encoder();
    if (!encode) return fail(PS_ERR_CUDA, "the driver does not provide cuTensorMapEncodeTiled");
    const int Hq = a.shape.n_q_heads, G = Hq / a.shape.n_kv_heads, d = a.shape.head_dim;
    const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)Hq, (cuuint64_t)a.total_q};
    const cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)Hq * d * 2};
    const cuuint32_t box[3] = {64, (cuuint32_t)G, (cuuint32_t)(128 / G)};
    const cuuint32_t elem_strides[3] = {1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(a.q), dims, strides, box,
                              elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(PS_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return PS_OK;
}

ps_status encode_pool_map(const RunArgs& a, CUtensorMap* map) {
    EncodeTiledFn encode = tensor_map_encoder();
    if (!encode) return fail(PS_ERR_CUDA, "the driver does not provide cuTensorMapEncodeTiled");
    const cuuint64_t dims[2] = {kPoolBlock / 8, (cuuint64_t)a.num_pages * a.shape.n_kv_heads * (a.shape.head_dim / 32)};
    const cuuint64_t strides[1] = {kPoolBlock};
    const cuuint32_t box[2] = {kPoolBlock / 8, 1};
    const cuuint32_t elem_strides[2] = {1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<char*>(a.pool), dims, strides, box, elem_strides,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(PS_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return PS_OK;
}

ps_status launch_prefill_pair(const RunArgs& a) {
    static PerDeviceOnce configured;
    const ps_status cfg = once_per_device(configured, []() -> ps_status {
        PS_CUDA_TRY(cudaFuncSetAttribute(prefill_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
        return PS_OK;
    });
    if (cfg != PS_OK) return cfg;
    PairParams p;
    p.pool = a.pool;
    p.num_pages = a.num_pages;
    p.block_table = a.block_table;
    p.max_pages = a.max_pages;
    p.out = a.out;
    p.lse = a.lse;
    p.hdr = a.w.hdr;
    p.items = a.w.prefill;
    p.n_items = a.w.n_prefill;
    p.pair_start = a.w.n_prefill_ctas > 0 ? a.w.prefill_cta_start : nullptr;
    p.part_lse = a.w.part_lse;
    p.part_o = a.w.part_o;
    p.Hq = a.shape.n_q_heads;
    p.Hkv = a.shape.n_kv_heads;
    p.G = p.Hq / p.Hkv;
    p.n_req = a.n_req;
    p.total_q = a.total_q;
    p.n_part_slots = (int32_t)a.w.n_part_slots;
    p.wait_limit_ns = (uint32_t)a.wait_limit_ns;
    p.tag = a.tag;
    p.flags = ((uintptr_t)a.out % 32 == 0 ? kOutAligned32 : 0) | (a.inline_items ? kInlineList : 0) | (a.beside ? kBeside : 0);
    InlineItems inl;
    fill_inline_items(a, inl);
    CUtensorMap q_map;
    const ps_status enc = encode_q_map(a, &q_map);
    if (enc != PS_OK) return enc;
    CUtensorMap pool_map;
    const ps_status enc_pool = encode_pool_map(a, &pool_map);
    if (enc_pool != PS_OK) return enc_pool;
    const int pairs = a.w.n_prefill_ctas > 0 ? a.w.n_prefill_ctas : (a.w.n_prefill < a.pf_sms / 2 ? a.w.n_prefill : (a.pf_sms > 1 ? a.pf_sms / 2 : 1));
    return launch_kernel(prefill_pair_kernel, 2 * pairs, kThreads, kSmemBytes, a.stream, 2, a.early, p, q_map, pool_map, inl);
}

}  // namespace ps
