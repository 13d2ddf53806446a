// Prefill-chunk attention for head dimension 64: a CTA per item.
//
// A chunk's rows attend the prior context plus the chunk's own earlier tokens (paper sections 2.4 and 4.7).  An item = up to
// two consecutive q tiles (A, B) of 128 (token, head) rows -- the G heads that share a kv head x 128 / G tokens -- over one key
// range; both consume the same K and V tiles of 128 keys.  At this head dimension a score costs the tensor core half of what
// it costs at 128 and the exp2 unit as much, so that unit is the bound: 1024 cycles a tile of 128 x 128 scores.  Hence
// everything is arranged for the softmax warps never to wait:
//
//   warps 0-7   softmax of q tile A, warps 8-15 of B: thread = half a row (64 of a tile's 128 keys)
//   warp 16     producer: K and V tiles (gathered pool blocks), Q
//   warp 17     issues the MMAs of A: QK^T (M 128, N 128, both operands in shared memory), PV (M 128, N 64, weights in tensor memory)
//   warp 18     those of B
//   warp 19     fetches the CTA's items ahead of their use
//
// TMEM columns: scores of A and B at 0 and 128, weights (bf16) at 256 and 320, O at 384 and 448.  A softmax warp loads all of its
// scores before it computes, so QK^T of the next key tile is issued while they are being worked on and its scores are there
// when they are done; PV of one tile runs under the softmax of the next.  Weights are relative to a sample of the row's own
// scores instead of a running maximum, with rows whose sums leave the range run again, as in prefill_pair.cu.
//
// What bounds it: a 128-key step of both q tiles takes some 2700 cycles, of which the exp2 unit needs 2048.  An mbarrier's answer takes
// a warp some 400 cycles beside those exponentials, whatever it is; so each q tile has an MMA warp of its own, which asks three
// things a step (K and V land on one barrier, and it is asked together with the scores').
// Measured (B200, N(0,1) data, kernel alone), before (two score tiles, a running maximum, one MMA warp) -> with one MMA warp and
// the scores of three tiles in turn, weights over them -> with two MMA warps and weights apart -> now:
//     8 q / 8 kv heads, 2048 tokens on 8192  72.6 -> 70.3 -> 61.4 -> 60.4 us      16 / 2  129.5 -> 123.6 -> 108.2 -> 105.9
//     two chunks of 768 and 1224 on 3600     44.7 -> 42.6 -> 38.4 -> 38.3;  48 decode rows beside them, whole iteration, 65.9 -> 63.1
// A chunk of 32 tokens on 100 takes 8.7 us instead of 11.3 (launch included).
// The time depends on the data: an item with a row whose scores lie some 69 above its sample's runs three times.  With N(0, 1) keys
// (whole run with append, 8/8 and 16/2 heads): 2048 tokens on 8192 64 and 111 us up to scores of standard deviation 8, and 16 at 8/8, 160
// and 289 from 24 on (with a running maximum, as before, 82 and 145); fresh prompts of 900 to 2000 tokens 35 and 46 up to 16, 83 and 112 from
// 24 on (49 and 55).
#include "tcgen05.cuh"

namespace ps {

namespace {

constexpr int kThreads = 640;
constexpr int kProducerWarp = 16, kMmaWarp = 17, kItemWarp = 19;  // (MMA warps: 17 of A, 18 of B)
constexpr int kRegsSoftmax = 104, kRegsOther = 64;  // 640 x 96 at launch = 512 x 104 + 128 x 64
constexpr int D = 64;
constexpr int kTileKeys = 128;
constexpr int kRows = 128;  // of a q tile
constexpr float kScaleLog2 = scale_log2(D);
constexpr float kSumMin = 8.7e-19f, kSumMax = 1.26e30f;  // 2^-60, 2^100: row sums outside are recomputed (prefill_pair.cu)
constexpr int kStages = 4;       // of K, and of V
constexpr int kTileBytes = 128 * 128;  // a Q, K or V tile: 128 rows of 64 elements
constexpr int kOffQ = 0;               // two buffers of tiles A, B
constexpr int kOffK = kOffQ + 4 * kTileBytes;
constexpr int kOffV = kOffK + kStages * kTileBytes;
constexpr int kOffBar = kOffV + kStages * kTileBytes;
constexpr int kItemRing = 8;
constexpr int kAheadTiles = 12;        // key tiles of items fetched ahead
constexpr int kRingConsumers = 19;     // every warp but the one that fetches them
constexpr uint32_t kColP = 256, kColO = 384;  // (S at 0)

struct Bars {  // byte offsets from the barrier block
    static constexpr int kv_full = 0, q_full = kv_full + 8 * kStages;
    static constexpr int kv_empty = q_full + 16, q_empty = kv_empty + 8 * kStages;  // either q tile's MMAs that read it have retired
    // per q tile: scores there, loaded by the softmax warps; weights there, read by PV; O there.  (Its softmax warps have read O
    // when they have the next item's first weights ready.)
    static constexpr int s_full = q_empty + 16, s_free = s_full + 16, p_ready = s_free + 16, p_free = p_ready + 16, o_done = p_free + 16;
    static constexpr int mma_drained = o_done + 16;       // both MMA warps'
    static constexpr int item_full = mma_drained + 8, item_empty = item_full + 8 * kItemRing;
    static constexpr int n_bars = (item_empty + 8 * kItemRing) / 8;
    static constexpr int tmem_slot = item_empty + 8 * kItemRing, abort_slot = tmem_slot + 4, limit_slot = abort_slot + 4;
    static constexpr int armed = limit_slot + 4;                     // parity of the last phase armed with copies: stages, Q buffers
    static constexpr int n_armed = kStages + 2;
    static constexpr int again = armed + 4 * n_armed;                // per ring slot a byte per q tile and quarter of its rows: sums out of range
    static constexpr int ring = (again + 8 * kItemRing + 15) / 16 * 16;
    static constexpr int redo = ring + kItemRing * (int)sizeof(PrefillItem);      // records to run again
    static constexpr int row_part = redo + kItemRing * (int)sizeof(PrefillItem);  // [q tile's item & 3][softmax warpgroup] per row: (sum or maximum, that number in the low byte of the sum's rounding)
    static constexpr int bytes = row_part + 16 * kRows * 8;
};
constexpr int kSmemBytes = kOffBar + Bars::bytes + 1024;  // + alignment slack
static_assert(kSmemBytes <= 232448 && Bars::armed % 4 == 0 && sizeof(PrefillItem) == 32, "shared memory");
static_assert(kPrefillRowsPerItem == 2 * kRows, "an item is two q tiles");
// How a record's item is run (in bits 24 up of n_tok): prefill_pair.cu
constexpr uint32_t kModePlain = 0, kModeMax = 1, kModeRelative = 2;

struct Params {
    const int32_t* block_table;
    __nv_bfloat16* out;
    float* lse;
    WsHeader* hdr;
    const PrefillItem* items;
    const int32_t* cta_start;  // static partition: CTA b runs items [cta_start[b], cta_start[b + 1]); null = dynamic queue
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
static_assert(sizeof(Params) <= 128, "parameter block");

__global__ void __launch_bounds__(kThreads, 1) prefill_d64_kernel(const Params p, const __grid_constant__ CUtensorMap q_map,
                                                                   const __grid_constant__ CUtensorMap pool_map, const __grid_constant__ InlineItems inl) {
    extern __shared__ char smem_raw[];
    char* smem = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + kOffBar;
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + kOffBar + Bars::abort_slot);
    volatile int* const s_armed = reinterpret_cast<volatile int*>(smem + kOffBar + Bars::armed);  // (-1: never; read only after an abort)
    // (through a shuffle, so that the compiler knows it to be warp-uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        s_abort[0] = 0;
        s_abort[1] = (int)p.wait_limit_ns;
    }
    if (warp == 0) {
        tmem_alloc(bars + Bars::tmem_slot, 512);
        tmem_relinquish();
    }
    const int tile_tok = kRows / p.G;
    const int g_shift = 31 - __clz(p.G);  // G is a power of two
    volatile uint8_t* const again = reinterpret_cast<volatile uint8_t*>(smem + kOffBar + Bars::again);
    uint4* const ring = reinterpret_cast<uint4*>(smem + kOffBar + Bars::ring);  // two uint4 per record
    uint4* const redo = reinterpret_cast<uint4*>(smem + kOffBar + Bars::redo);
    // next item of this CTA's static share, or of the queue all CTAs of the run drain
    const bool inline_list = (p.flags & kInlineList) != 0, static_share = inline_list || p.cta_start != nullptr;
    auto next_item = [&](int cur, int end) { return static_share ? (cur < end ? cur : p.n_items) : atomicAdd(&p.hdr->prefill_next, 1); };
    auto start_of = [&](int cta) { return inline_list ? inl.start[cta] : __ldg(p.cta_start + cta); };
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
    if (threadIdx.x == kItemWarp * 32) {
        // the first item's record is on its way before the roles begin
        const int idx = next_item(static_share ? start_of(blockIdx.x) : 0, static_share ? start_of(blockIdx.x + 1) : 0);
        uint4 a = make_uint4(0, 0, 0, 0), b = a;
        if (idx < p.n_items) record(idx, a, b);
        redo[0] = a;
        redo[1] = b;
    }
    for (int k = threadIdx.x; k < Bars::n_bars; k += kThreads) {
        const int off = 8 * k;
        uint32_t count = 1;
        if (off >= Bars::kv_empty && off < Bars::s_full) count = 2;
        else if (off >= Bars::s_free && off < Bars::p_free) count = 8;
        else if (off == Bars::mma_drained) count = 2;
        else if (off >= Bars::item_empty) count = kRingConsumers;
        mbar_init(bars + off, count);
        mbar_fence_init();
    }
    for (int k = threadIdx.x; k < 16 * kRows; k += kThreads) store_tagged(bars + Bars::row_part + 8 * k, 0.f, 0xffffffffu);
    if (threadIdx.x < 8 * kItemRing) again[threadIdx.x] = 0;
    if (threadIdx.x < Bars::n_armed) s_armed[threadIdx.x] = -1;
    if (!(p.flags & kBeside)) pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t*>(smem + kOffBar + Bars::tmem_slot), 0);
    // warp-uniform result, so that the warp-collective instructions that follow stay converged
    auto wait_all = [](uint32_t bar, uint32_t parity, volatile int* abort_flag) {
        return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag));
    };
    constexpr uint32_t kIdescQK = instr_desc(kRows, kTileKeys, false);
    constexpr uint32_t kIdescPV = instr_desc(kRows, D, true);
    // Consumer side of the record ring: record number n; false at the end-of-work record or on abort.  A softmax warp gives the
    // slot back when its part of the item's sums has been checked, so that a free slot means a checked item.
    auto take_record = [&](uint32_t n, uint4& a, uint4& b, bool give_back) -> bool {
        const uint32_t slot = n % kItemRing;
        if (!wait_all(bars + Bars::item_full + 8 * slot, (n / kItemRing) & 1, s_abort)) return false;
        a = ring[2 * slot];
        b = ring[2 * slot + 1];
        __syncwarp();
        if (give_back && lane == 0) mbar_arrive(bars + Bars::item_empty + 8 * slot);
        return (int32_t)b.y > 0;
    };
    auto tiles_of = [](const uint4& a) { return ((int32_t)a.w - (int32_t)a.z + kTileKeys - 1) / kTileKeys; };
    // Key tiles of q tile A: with a second q tile they may be fewer, by those that only B's rows see; one at least, which leaves
    // rows that see nothing of the item's key range with empty sums.
    auto tiles_of_a = [&](const uint4& a, const uint4& b) {
        if ((int)(b.y & 0xffffu) <= tile_tok) return tiles_of(a);
        return max(1, (min((int)a.w, (int)b.w + tile_tok) - (int)a.z + kTileKeys - 1) / kTileKeys);
    };

    if (warp < 16) {
        // ====================================================================
        // softmax: warpgroup 2 x + h takes keys 64 h .. 64 h + 63 of the key tiles of q tile x; thread t owns row t
        // ====================================================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
        const uint32_t x = warp >> 3, h = (warp >> 2) & 1;
        const int t = threadIdx.x & 127;
        const uint32_t lane_tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        auto row_part = [&](uint32_t item, uint32_t half) { return bars + Bars::row_part + 8 * (((item & 3) * 4 + 2 * x + half) * kRows + t); };
        // the other half's entry for this row, once it carries `item`'s number
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
        const uint32_t s_addr = lane_tm + x * 128 + h * 64, p_addr = lane_tm + kColP + x * 64 + h * 32;
        uint32_t n_item = 0, v_tiles = 0;  // v_tiles: number of the item's first key tile
        uint32_t mine = 0, items_x = 0;    // score tiles and items of this q tile
        bool ok = true;
        while (ok) {
            uint4 ra, rb;
            if (!take_record(n_item, ra, rb, false)) break;
            const int key_begin = (int)ra.z, key_end = (int)ra.w, n_tok = (int)(rb.y & 0xffffu), first_pos = (int)rb.w;
            const uint32_t mode = rb.y >> 24;
            const bool two = n_tok > tile_tok;
            const int n_a = tiles_of_a(ra, rb), n_b = two ? tiles_of(ra) : 0, n_tiles = x ? n_b : n_a;
            auto give_back = [&]() {
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + Bars::item_empty + 8 * (n_item % kItemRing));
            };
            if (n_tiles == 0) {  // no tile B
                give_back();
                v_tiles += n_a;
                ++n_item;
                continue;
            }
            const int i = (int)x * tile_tok + (t >> g_shift);  // token of this row within the item
            const int limit = min(first_pos + i + 1, key_end);  // first key this row does not see
            const int plain_keys = min(first_pos + (int)x * tile_tok + 1, key_end);  // keys that every row of this q tile sees
            float rounding = 0.f;      // what rounding the weights has added to l
            float ref = 0.f, l = 0.f;  // l: sum of this thread's weights (or their maximum)
            float top = -INFINITY;     // largest score of its halves that needed no mask
            if (mode == kModeRelative) {
                ref = -INFINITY;
                for (uint32_t hf = 0; hf < 2 && ok; ++hf) {
                    float m, unused;
                    ok = read_tagged(row_part(items_x - 1, hf), items_x - 1, m, unused);
                    ref = fmaxf(ref, m);
                }
                if (!ok) break;
                if (ref == -INFINITY) ref = 0.f;
            }
            if (mode == kModeMax) l = -INFINITY;
            for (int j = 0; j < n_tiles; ++j) {
                const uint32_t par = (mine + (uint32_t)j) & 1;
                ok = wait_all(bars + Bars::s_full + 8 * x, par, s_abort);
                if (!ok) break;
                tc_fence_after();
                if (j == 0 && mode == kModePlain) {
                    // The row's reference, the same in both halves.
                    uint32_t sv[32];
                    tmem_ld32(lane_tm + x * 128 + 32, sv);
                    tmem_wait_ld();
                    float mx = -INFINITY;
#pragma unroll
                    for (int c = 0; c < 32; c += 2) mx = max3(mx, __uint_as_float(sv[c]), __uint_as_float(sv[c + 1]));
                    // (rows that see fewer than 64 keys: below)
                    if (limit - key_begin >= 64 && fabsf(mx) < INFINITY) ref = mx * kScaleLog2;
                }
                const int tile_base = key_begin + j * kTileKeys;
                const int vis = limit - tile_base - (int)h * 64;  // columns [0, vis) of this half are visible to this row
                // columns of this half that every row of the warp sees (later rows see no fewer)
                const int vis_all = tile_base + kTileKeys <= plain_keys ? 64 : __shfl_sync(0xffffffffu, vis, 0);
                if (mode != kModeMax && vis_all >= 64) {
                    uint32_t s0[32], s1[32], packed[32];
                    tmem_ld32(s_addr, s0);
                    tmem_ld32(s_addr + 32, s1);
                    tmem_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bars + Bars::s_free + 8 * x, lane == 0);
                    uint64_t ls0 = 0ull, ls1 = 0ull;
                    weights32<D>(s0, ref, ls0, ls1, top, packed);
                    weights32<D>(s1, ref, ls0, ls1, top, packed + 16);
                    ok = wait_all(bars + Bars::p_free + 8 * x, par ^ 1, s_abort);  // the tile before's weights have been read
                    if (!ok) break;
                    tc_fence_after();
                    tmem_st32(p_addr, packed);
                    float a0, a1, a2, a3;
                    unpack2(ls0, a0, a1);
                    unpack2(ls1, a2, a3);
                    l += (a0 + a2) + (a1 + a3);
                } else {
                    // Diagonal and ragged halves, the only ones of rows with few visible keys.
                    const int vis_any = __shfl_sync(0xffffffffu, vis, 31);  // columns that some row of the warp sees
                    ok = wait_all(bars + Bars::p_free + 8 * x, par ^ 1, s_abort);
                    if (!ok) break;
                    tc_fence_after();
                    if (mode == kModePlain && j == 0 && h == 0 && __any_sync(0xffffffffu, vis < 64)) {
                        // Rows that see fewer than 64 keys of the item, all of them here: relative to their maximum, so that the
                        // weight that counts most is 1 and rounds to itself.  (This thread also writes their log-sum-exp.)
                        const float mx = masked_max64(s_addr, vis, vis_any);
                        if (vis < 64 && mx > -INFINITY) ref = mx * kScaleLog2;
                    }
                    if (mode == kModeMax) l = fmaxf(l, masked_max64(s_addr, vis, vis_any) * kScaleLog2);
                    else masked_weights64<D>(s_addr, p_addr, vis, vis_any, ref, l, rounding);
                    tc_fence_before();
                    __syncwarp();
                    mbar_arrive_if(bars + Bars::s_free + 8 * x, lane == 0);
                }
                // keys at or past key_end: their V rows may be stale or poisoned; zero them (for this q tile's PV: the other's
                // softmax does as much) so that 0 * V = 0
                const int n_keys = key_end - tile_base;
                if (n_keys < kTileKeys && h == 0) {
                    const uint32_t vt = v_tiles + (uint32_t)j, s = vt % kStages;
                    ok = wait_all(bars + Bars::kv_full + 8 * s, (vt / kStages) & 1, s_abort);
                    if (!ok) break;
                    if (t >= n_keys) {
                        char* vrow = smem + kOffV + s * kTileBytes + t * 128;
#pragma unroll
                        for (int u = 0; u < 8; ++u) *reinterpret_cast<uint4*>(vrow + u * 16) = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                mbar_arrive_if(bars + Bars::p_ready + 8 * x, lane == 0);
            }
            if (!ok) break;
            // ---- end of the item: the halves' sums, then the output, 32 columns each ----
            if (mode != kModeMax) {
                // PV multiplies rounded weights, and their sum is what normalises the output: counted for the largest weight of
                // each of a row's two threads (prefill_pair.cu)
                const float e = fast_exp2(fmaf(top, kScaleLog2, -ref)), d = bf16_lo(pack_bf16(e, 0.f)) - e;
                l += d;
                rounding += d;
            }
            store_tagged(row_part(items_x, h), l, (items_x & 0xffu) | (__float_as_uint(rounding) & ~0xffu));
            rounding = __uint_as_float(__float_as_uint(rounding) & ~0xffu);  // (as the other half reads it)
            float lp, rp;
            ok = read_tagged(row_part(items_x, h ^ 1), items_x, lp, rp);
            if (!ok) break;
            l += lp;
            rounding += rp;
            const float inv = l > 0.f ? 1.f / l : 0.f;
            const float lse_v = l > 0.f ? (ref + log2f(l - rounding)) * 0.6931471805599453f : -INFINITY;
            // (a row that sees no key of this item's range has an empty sum)
            const bool bad = i < n_tok && limit > key_begin && !(l >= kSumMin && l <= kSumMax);
            const uint32_t quarter = x * 4 + (warp & 3);
            bool write = mode == kModeRelative ? ((rb.y >> (16 + quarter)) & 1u) != 0 : mode == kModePlain;
            if (mode == kModePlain && __any_sync(0xffffffffu, bad)) {
                if (lane == 0) again[8 * (n_item % kItemRing) + quarter] = 1;
                write = false;
            }
            give_back();
            const bool valid = i < n_tok && write;
            const int q_tok = (int)rb.x, part_slot = (int)rb.z, kv_head = (int)ra.y;
            const int64_t orow = (int64_t)(q_tok + i) * p.Hq + kv_head * p.G + (t & (p.G - 1));
            const int64_t prow = (int64_t)part_slot + (int64_t)x * kRows + t;
            ok = wait_all(bars + Bars::o_done + 8 * x, items_x & 1, s_abort);
            if (!ok) break;
            tc_fence_after();
            uint32_t v[32];
            tmem_ld32(lane_tm + kColO + x * D + h * 32, v);
            tmem_wait_ld();
            tc_fence_before();
            // Every lane writes its own row, 32 bytes (a DRAM sector) at a time.
            if (valid) {
                if (part_slot < 0) {
                    char* dst = reinterpret_cast<char*>(p.out + orow * D + h * 32);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        uint32_t y[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) y[c] = pack_bf16(__uint_as_float(v[u * 16 + 2 * c]) * inv, __uint_as_float(v[u * 16 + 2 * c + 1]) * inv);
                        store32(dst + 32 * u, y, p.flags & kOutAligned32);
                    }
                } else {
                    char* dst = reinterpret_cast<char*>(p.part_o + prow * D + h * 32);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        uint32_t y[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) y[c] = __float_as_uint(__uint_as_float(v[u * 8 + c]) * inv);
                        store32(dst + 32 * u, y, true);
                    }
                }
            }
            if (valid && h == 0) {
                if (part_slot >= 0) p.part_lse[prow] = lse_v;
                else if (p.lse) p.lse[orow] = lse_v;
            }
            mine += n_tiles;
            v_tiles += tiles_of(ra);
            ++items_x;
            ++n_item;
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
        if (warp == kProducerWarp) {
            // ================================================================
            // producer: K tiles, V tiles, Q.  K/V tiles of a chunk's sequence are read again by every other item of that sequence:
            // they are marked last to leave L2.
            // ================================================================
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
                // Pool rows (2 KB blocks: K and V of a page) of four tiles at a time, one page per lane, requested four tiles
                // ahead; -8 for a page that is not there.
                auto pool_row = [&](int page, int idx) {
                    const bool has = idx < n_pages, good = has && (uint32_t)page < (uint64_t)p.num_pages;
                    if (has && !good) report(p.hdr, p.tag, kStatusBounds);
                    return good ? (page * p.Hkv + kv_head) * 2 : -8;
                };
                int row = -8, bt_next = lane < n_pages ? __ldg(bt + lane) : 0;
                for (int j = 0; j < n_tiles; ++j, ++tc) {
                    if ((j & 3) == 0) {
                        row = pool_row(bt_next, j * 8 + lane);
                        bt_next = (j + 4) * 8 + lane < n_pages ? __ldg(bt + (j + 4) * 8 + lane) : 0;
                    }
                    int r[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) r[k] = __shfl_sync(0xffffffffu, row, (j & 3) * 8 + k);
                    const uint32_t s = tc % kStages, par = (tc / kStages) & 1;
                    ok = wait_all(bars + Bars::kv_empty + 8 * s, par ^ 1, s_abort);
                    if (!ok) break;
                    if (elect_one()) {
                        const uint32_t land = bars + Bars::kv_full + 8 * s, k = sbase + kOffK + s * kTileBytes, v = sbase + kOffV + s * kTileBytes;
                        mbar_expect_tx(land, 2 * kTileBytes);
                        s_armed[s] = (int)par;
                        gather4(k, &pool_map, r[0], r[1], r[2], r[3], land, kv_policy);
                        gather4(k + 4 * kPoolBlock, &pool_map, r[4], r[5], r[6], r[7], land, kv_policy);
                        gather4(v, &pool_map, r[0] + 1, r[1] + 1, r[2] + 1, r[3] + 1, land, kv_policy);
                        gather4(v + 4 * kPoolBlock, &pool_map, r[4] + 1, r[5] + 1, r[6] + 1, r[7] + 1, land, kv_policy);
                    }
                    __syncwarp();
                    if (j == 0) {
                        // Q tiles: rows (token, head of the group) in token-major order, one box of [128 / G tokens][G heads][64
                        // elements] each, in the 128-byte swizzle
                        const uint32_t qb = n_item & 1, qpar = (n_item >> 1) & 1;
                        const int n_x = (int)(rb.y & 0xffffu) > tile_tok ? 2 : 1;
                        ok = wait_all(bars + Bars::q_empty + 8 * qb, qpar ^ 1, s_abort);
                        if (!ok) break;
                        if (lane == 0) {
                            mbar_expect_tx(bars + Bars::q_full + 8 * qb, n_x * kTileBytes);
                            s_armed[kStages + qb] = (int)qpar;
                            for (int x = 0; x < n_x; ++x)
                                tma_load_3d(sbase + kOffQ + (2 * qb + x) * kTileBytes, &q_map, 0, kv_head * p.G, (int32_t)rb.x + x * tile_tok,
                                            bars + Bars::q_full + 8 * qb);
                        }
                        __syncwarp();
                    }
                }
            }
        } else if (warp == kMmaWarp || warp == kMmaWarp + 1) {
            // ================================================================
            // MMA issue for q tile x: QK^T of a key tile once the scores of the one before have been loaded, PV of a tile once its
            // weights are there.  A stage's barriers count both q tiles: one that has no rows for a key tile passes it over.
            // ================================================================
            const uint32_t x = warp - kMmaWarp;
            const uint64_t desc_k = smem_desc(0, 16, 1024);
            const uint64_t desc_v = smem_desc(0, kTileBytes, 1024);
            const uint32_t q_lo = (sbase + kOffQ) >> 4, k_lo = (sbase + kOffK) >> 4, v_lo = (sbase + kOffV) >> 4;
            const uint32_t hi_k = (uint32_t)(desc_k >> 32), hi_v = (uint32_t)(desc_v >> 32);
            const uint32_t s_tm = tmem + x * 128, p_tm = tmem + kColP + x * 64, o_tm = tmem + kColO + x * D;
            uint32_t n_item = 0, n_qk = 0, n_pv = 0;  // items begun, QK^Ts and PVs issued
            uint32_t k_tc = 0, v_tc = 0;                          // key tiles that either has reached
            uint32_t qb = 0;
            int j = 0, n_mine = 0, n_all = 0;  // of the item whose QK^T is being issued: its next key tile, this q tile's, all
            uint32_t flags = 0;                // of the tiles whose PV is outstanding, eight bits each: first, last, key tiles to pass over then
            bool ok = true, more = true, in_item = false;
            auto pass = [&]() {
                ok = wait_all(bars + Bars::kv_full + 8 * (v_tc % kStages), (v_tc / kStages) & 1, s_abort);
                if (ok && lane == 0) mbar_arrive(bars + Bars::kv_empty + 8 * (v_tc % kStages));
                ++v_tc;
            };
            while (true) {
                if (more && n_qk - n_pv < 2) {
                    if (!in_item) {
                        // (with a PV outstanding the next record is not waited for)
                        if (n_qk != n_pv && !__all_sync(0xffffffffu, mbar_test_wait(bars + Bars::item_full + 8 * (n_item % kItemRing), (n_item / kItemRing) & 1)))
                            goto issue_pv;
                        uint4 ra, rb;
                        // (an item without rows of this q tile is taken when no PV is outstanding)
                        const uint32_t slot = n_item % kItemRing;
                        if (x == 1 && n_qk != n_pv && __all_sync(0xffffffffu, (int)(ring[2 * slot + 1].y & 0xffffu) <= tile_tok)) goto issue_pv;
                        more = take_record(n_item, ra, rb, true);
                        if (!more) continue;
                        const bool two = (int)(rb.y & 0xffffu) > tile_tok;
                        n_all = __shfl_sync(0xffffffffu, tiles_of(ra), 0);
                        n_mine = __shfl_sync(0xffffffffu, x == 0 ? tiles_of_a(ra, rb) : two ? n_all : 0, 0);
                        qb = n_item & 1;
                        ok = wait_all(bars + Bars::q_full + 8 * qb, (n_item >> 1) & 1, s_abort);
                        if (!ok) break;
                        ++n_item;
                        j = 0;
                        if (n_mine == 0) {
                            if (lane == 0) mbar_arrive(bars + Bars::q_empty + 8 * qb);
                            for (int k = 0; k < n_all && ok; ++k) pass();
                            k_tc = v_tc;
                            if (!ok) break;
                            continue;
                        }
                        in_item = true;
                    }
                    const uint32_t ks = k_tc % kStages;
                    // (Asked for together: an answer takes some 400 cycles, because the question queues behind the softmax warps'
                    // exponentials.  K and V land on one barrier for the same reason.)
                    const bool there = mbar_test_wait(bars + Bars::kv_full + 8 * ks, (k_tc / kStages) & 1), loaded = mbar_test_wait(bars + Bars::s_free + 8 * x, (n_qk & 1) ^ 1);
                    if (!__all_sync(0xffffffffu, there && loaded)) {
                        ok = wait_all(bars + Bars::kv_full + 8 * ks, (k_tc / kStages) & 1, s_abort);
                        if (ok) ok = wait_all(bars + Bars::s_free + 8 * x, (n_qk & 1) ^ 1, s_abort);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const bool last = j + 1 == n_mine;
                    if (elect_one()) {
                        const uint32_t q = (uint32_t)desc_k + q_lo + (2 * qb + x) * (kTileBytes >> 4), k = (uint32_t)desc_k + k_lo + ks * (kTileBytes >> 4);
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)
                            tc_mma_ss(s_tm, desc64(q + kk * (32 >> 4), hi_k), desc64(k + kk * (32 >> 4), hi_k), kIdescQK, kk > 0);
                        tc_commit(bars + Bars::s_full + 8 * x);
                        if (last) tc_commit(bars + Bars::q_empty + 8 * qb);
                    }
                    __syncwarp();
                    flags |= ((j == 0 ? 1u : 0u) | (last ? 2u | (uint32_t)(n_all - n_mine) << 2 : 0u)) << (8 * (n_qk - n_pv));
                    k_tc += last ? n_all - j : 1;
                    ++n_qk;
                    ++j;
                    in_item = !last;
                    if (n_qk - n_pv < 2) continue;
                }
            issue_pv:
                if (n_qk == n_pv) break;
                const uint32_t vs = v_tc % kStages;
                const bool first = flags & 1u, last = flags & 2u;
                ok = wait_all(bars + Bars::p_ready + 8 * x, n_pv & 1, s_abort);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t v = (uint32_t)desc_v + v_lo + vs * (kTileBytes >> 4);
#pragma unroll
                    for (int kk = 0; kk < kTileKeys / 16; ++kk)
                        tc_mma_ts(o_tm, p_tm + kk * 8, desc64(v + kk * (2048 >> 4), hi_v), kIdescPV, (!first || kk > 0) ? 1u : 0u);
                    tc_commit(bars + Bars::p_free + 8 * x);
                    tc_commit(bars + Bars::kv_empty + 8 * vs);
                    if (last) tc_commit(bars + Bars::o_done + 8 * x);
                }
                __syncwarp();
                ++v_tc;
                ++n_pv;
                for (uint32_t k = flags >> 2 & 63u; k > 0 && ok; --k) pass();
                if (!ok) break;
                flags >>= 8;
            }
        } else {
            // ================================================================
            // items: fetches the CTA's records, from its static share or the queue, and puts them into the ring as slots come free
            // ================================================================
            int static_cur = 0, static_end = 0;
            if (static_share) {
                static_cur = start_of(blockIdx.x) + 1;
                static_end = start_of(blockIdx.x + 1);
            }
            uint32_t mode = kModePlain, redo_head = 0, redo_tail = 0;  // records put aside
            uint4 fa = redo[0], fb = redo[1];                          // the record fetched; n_tok = 0: end of work
            uint4 na, nb;                                              // the record published last
            __syncwarp();  // (the ring of records put aside begins with the first one's place)
            auto check_record = [&]() {
                if ((int32_t)fb.y == 0) return;
                // A record that points outside the batch (only a damaged work list has one) ends this CTA's work and
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
                }
                __syncwarp();
                if (from_fetched && (int32_t)nb.y == 0) break;
                // An item taken early from the queue is one that an idle CTA cannot take: only one is, beyond kAheadTiles.  (And
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
    if (warp == kMmaWarp || warp == kMmaWarp + 1) {
        if (elect_one()) tc_commit(bars + Bars::mma_drained);
        __syncwarp();
        mbar_wait(bars + Bars::mma_drained, 0, kDrainLimitNs);
    }
    tc_fence_before();
    __syncthreads();  // every role has left its loop
    if (*s_abort) {
        // A bounded wait ran out somewhere in this CTA: the output is invalid and the run is flagged.  Before the CTA gives back
        // its shared and tensor memory, the copies requested get a bounded time to land (the MMAs have retired).
        if (threadIdx.x == 0) report(p.hdr, p.tag, kStatusTimeout);
        if (warp == kProducerWarp) {
            const uint64_t t0 = global_timer_ns();
            for (int k = 0; k < Bars::n_armed; ++k) {
                const int par = s_armed[k];
                const int64_t left = kDrainLimitNs - (int64_t)(global_timer_ns() - t0);
                const int bar = k < kStages ? Bars::kv_full + 8 * k : Bars::q_full + 8 * (k - kStages);
                if (par >= 0) mbar_wait(bars + bar, (uint32_t)par, left);
            }
        }
        __syncthreads();
    }
    if (warp == 0) tmem_dealloc(tmem, 512);
    if ((p.flags & kBeside) && blockIdx.x == 0) pdl_wait();  // this kernel's end also means that of the decode kernel beside it
}

}  // namespace

ps_status launch_prefill_d64(const RunArgs& a) {
    static PerDeviceOnce configured;
    const ps_status cfg = once_per_device(configured, []() -> ps_status {
        PS_CUDA_TRY(cudaFuncSetAttribute(prefill_d64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
        return PS_OK;
    });
    if (cfg != PS_OK) return cfg;
    Params p;
    p.num_pages = a.num_pages;
    p.block_table = a.block_table;
    p.max_pages = a.max_pages;
    p.out = a.out;
    p.lse = a.lse;
    p.hdr = a.w.hdr;
    p.items = a.w.prefill;
    p.n_items = a.w.n_prefill;
    p.cta_start = a.w.n_prefill_ctas > 0 ? a.w.prefill_cta_start : nullptr;
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
    CUtensorMap q_map, pool_map;
    ps_status st = encode_q_map(a, &q_map);
    if (st == PS_OK) st = encode_pool_map(a, &pool_map);
    if (st != PS_OK) return st;
    const int grid = a.w.n_prefill_ctas > 0 ? a.w.n_prefill_ctas : (a.w.n_prefill < a.pf_sms ? a.w.n_prefill : a.pf_sms);
    return launch_kernel(prefill_d64_kernel, grid, kThreads, kSmemBytes, a.stream, 1, a.early, p, q_map, pool_map, inl);
}

}  // namespace ps
