// Host work partitioner and the per-iteration run entry point.
//
// The partition depends on the logical lengths only (never on page ids), so a
// batch produces the same items, the same summation order and therefore the
// same output bits under any assignment of physical pages.
#include <algorithm>
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <functional>
#include <iterator>
#include <atomic>
#include <mutex>
#include <new>
#include <unordered_map>
#include <utility>
#include <vector>

#include "common.cuh"

namespace ps {

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

constexpr int kDecodeUnitsPerWarp = 1;  // work units per resident warp (measured: 1 beats 2 and 3 on the decode-only batch)
// Smallest decode unit (pages) of a batch too small to give every warp its share: between 4 and 8, so that the
// longest row is cut into about 16 pieces at most.  Finer cuts spread a small batch over more warps (64 rows of
// 64 tokens: 13 us instead of 20; 8 rows of 512: 16 instead of 23), but every further piece of a row is one more
// partial result for the one warp that combines them (one row of 4096 tokens: 22 us at 32 pieces, 26 at 64).
constexpr int kDecodeMinPagesLo = 4, kDecodeMinPagesHi = 8, kDecodePiecesPerRow = 16;
// A CTA per piece (small batches): pages of a piece at most, and before a row is cut (8 and 4 for each of the 12 warps that a
// CTA has at head dimension 128, 4 and 2 for each of 24 at 64).
constexpr int kCtaMaxPiece = 96, kCtaMinPiece = 48;
constexpr int kPrefillKeyTile = 128;    // keys per tensor-core tile
// Measured on B200 (bandwidth against the number of SMs the decode kernel runs on), used with the prefill kernel's cost
// model to split the SMs of a mixed batch between the two kernels.
constexpr double kDecodePeakBytesPerSec = 6.7e12;
constexpr double kDecodeSharedPeakBytesPerSec = 6.0e12;  // decode rows beside a running prefill kernel
// Per SM with the memory system to itself, and 0.85 of it beside a prefill kernel: 16 to 48 SMs stream 130 GB/s each at head
// dimension 128 and 99 to 104 GB/s at 64.  (Less is taken at 64, where shares up to 92 SMs gain: 400 rows of 1000 tokens and a
// 1024-token chunk 148 us on 72 SMs, as 100 would have it, 144.5 on 84.)
static inline double decode_alone_rate_per_sm(const ps_shape& sh) { return sh.head_dim == 128 ? 135e9 : 88e9; }
static inline double decode_rate_per_sm(const ps_shape& sh) { return 0.85 * decode_alone_rate_per_sm(sh); }
constexpr double kKernelFloorSec = 12e-6;
// The merge kernel runs under the decode kernel where that is predicted to end this much after the prefill kernel (ps_attn_run()), with what
// a warp spends on each of its rows beside their pages, and on each segment of a row when it combines them.
constexpr double kMergeUnderDecodeSec = 2.5e-6, kRowSec = 2e-6, kSegmentSec = 0.09e-6;
constexpr double kDecodeManyBytes = 0.75e9;
constexpr int kDecodeAloneSms = 128;

// Cost model of a prefill kernel in units of one 128-key step of an item (256 rows): an item pays a fixed overhead
// (pipeline fill, output) plus one unit per key tile.
struct PrefillModel {
    double step_sec;      // SM-seconds of a step
    double fixed;         // steps an item costs beyond its key tiles
    double masked_extra;  // and the diagonal tile's slower softmax
    double cut;           // steps that cutting items costs: partial rows, merge kernel
    // Steps by which whole items may end later than an even split: what cutting costs a small batch, a kernel more and a list that has
    // to be uploaded.  Of up to kFewItems items, whose merge is quick; of more.
    double whole_few, whole;
    int sms_per_worker;   // an item is worked on by one CTA, or by a pair of them
};
// prefill.cu (fitted to per-CTA run times: 2.2 us per step, about 3 us per item, 1.2 us more for a masked tile).  Its items are never
// cut: `cut` is how far its queue ends behind an even split at most, for the shares of mixed batches.  (Without it, by the longest item
// alone: 239 rows of 359 tokens, 60 chunks of 24 and two of 953 and 555 102.7 -> 109.5 us, 40 rows of 2711 and 102 chunks 128.3 -> 135.9; 30
// drawn mixed batches of many short chunks, geometric mean 1.008.)
constexpr PrefillModel kSingleModel = {2.5e-6, 1.5, 0.5, 3.0, 0.0, 0.0, 1};
// prefill_pair.cu (72, 144 and 288 equal items on 74 pairs with 11 to 67 key tiles: 0.70 us per step of a pair, 2.8 us per
// item; the merge kernel takes about 8 us).  Cut instead of whole, a run with append, by the steps that whole items end later: 2 to 10
// items 12 steps 3 to 10 % longer, 14 steps 2 % shorter to 2 % longer, 16 steps 3 % shorter, 19 steps 8 %, 20 steps 13 to 17 % (24.9 -> 20.7 us);
// 16 items 16.5 steps 2 to 3 % longer, 18.8 steps the same; 24 items 17.9 steps 3 % longer, 19.6 steps 3 % shorter; 32 items 16 steps 12 %
// longer, 18.4 steps 2 %; 80 to 168 items 18.9 steps 2 % longer, 19.1 steps 1 % shorter.
constexpr int kFewItems = 12;
constexpr PrefillModel kPairModel = {1.45e-6, 3.5, 0.5, 9.0, 14.0, 18.5, 2};
// prefill_d64.cu (148 CTAs of 1 to 3 items of 6 to 29 key tiles, beside a decode kernel: 9.4 us a CTA, 3.1 an item, 1.28 a step; the
// merge kernel and the gap before it 7.5 us).  An item's 3.1 us are 2.4 steps; as 2, so that a smallest share holds two whole key tiles,
// 30 batches with cut items are 4 % faster: 256 tokens on 1500, 4 / 2 heads, 22.7 -> 20.4 us, 64 on 3000 18.3 -> 16.5, 700 and 300 on 1500
// at 8 / 8 26.4 -> 24.7.  Cut instead of whole, before that: 4 to 20 items 6.9 steps 1 to 40 % longer, 7.9 steps 8 % shorter to 12 % longer, 8.9
// steps 11 % shorter to 5 % longer; now with a line of 7.5 instead of 8 items of ten key tiles 3 to 12 % longer (1633 and 1051 fresh
// tokens beside 23 rows 29.5 -> 33.3) or 3 % shorter.
constexpr PrefillModel kD64Model = {1.28e-6, 1.5, 0.5, 6.0, 8.0, 8.0, 1};
// An item's cost at head dimension 64 as measured, by which the SMs of mixed batches are shared out.
static inline PrefillModel measured_model(const ps_shape& sh, PrefillModel m) {
    if (sh.head_dim == 64) m.fixed = 2.0, m.masked_extra = 0.4;
    return m;
}
// For plans that leave fewer partial rows, at the limit of the built-in scratch (ps_attn_plan()): items stay whole up to later ends, too.
static inline PrefillModel lean_model(const ps_shape& sh, PrefillModel m) {
    m.whole_few = m.whole = sh.head_dim == 64 ? 10.0 : 20.0;
    return measured_model(sh, m);
}
static inline const PrefillModel& prefill_model(const ps_shape& sh, bool pairs) { return sh.head_dim == 64 ? kD64Model : pairs ? kPairModel : kSingleModel; }
// Which kernel runs the prefill items.  Head dimension 64: a CTA per item.  128: a pair of CTAs, unless the items are short and
// there are enough for all SMs.  An item costs a CTA 3.5 us and 2.2 more a key tile, a pair 3.2 us and 0.73, so up to some
// four key tiles two items on two CTAs are done sooner; of few items a pair does each in less time.
// Measured (a run, us, single / pair): fresh prompts of 64 tokens 24 of them 19.4 / 23.5, 188 74 / 98; of 256 6 20.9 / 25.2,
// 24 48.5 / 61; of 512 6 35 / 42, 48 200 / 229; of 1024 12 151 / 148; 64 tokens on 192 40 times 45 / 34, 94 times 53 / 65; on
// 320 188 times 116 / 123; on 576 164 / 159.
static inline bool prefill_on_pairs(const ps_shape& sh, int num_sms, int64_t items, int64_t key_tiles) {
    const bool many = items >= 2.5 * num_sms && key_tiles <= 4.0 * items, some = items >= 1.25 * num_sms && key_tiles <= 1.75 * items;
    return sh.head_dim == 128 && !many && !some;
}

// A chunk of a few tokens runs as that many decode rows (token i of the chunk is a row that sees prior + i + 1 keys
// of the same sequence) instead of bringing in the prefill kernel for one small item: its launch and pipeline fill
// cost more than re-reading a short context a few times.  Bounded by the bytes the rows re-read, and only in batches
// whose decode rows are few: beside a long decode kernel the prefill kernel of a small chunk is hidden anyway.
// (measured: a 2-token chunk on 2048 tokens beside 8 decode rows of 512: 23.8 us instead of 29.8; 8 tokens on 900
// alone 16.4 instead of 22.6; 4 tokens on 1500 beside 128 rows of 2048 would be 169 instead of 165)
constexpr int kTinyChunkTokens = 8;
constexpr double kTinyChunkBytes = 32e6;
constexpr double kTinyChunkMaxDecodeBytes = 128e6;
static inline bool runs_as_decode(const ps_shape& sh, bool tiny_as_rows, int prior, int q_len) {
    if (q_len == 1) return true;
    if (!tiny_as_rows || q_len > kTinyChunkTokens) return false;
    return (double)q_len * ((double)prior + q_len) * 2.0 * sh.n_kv_heads * sh.head_dim * 2.0 <= kTinyChunkBytes;
}

}  // namespace ps

using namespace ps;

namespace {

// Which plan last put a work list into a given workspace.  Two plans that take turns on one workspace (or on the
// built-in scratch of ps_attn_run_static) each keep their own record of the slots they have used; a plan that finds
// another plan's serial here orders its upload behind everything already on the caller's stream instead of trusting
// that record.
std::mutex g_ws_mu;
std::unordered_map<const void*, uint64_t> g_ws_owner;
constexpr size_t kWsOwnerCap = 4096;  // forgetting an entry only costs its next run one stream fence

uint64_t next_plan_serial() {
    static std::atomic<uint64_t> next{1};
    return next.fetch_add(1, std::memory_order_relaxed);
}

// true if `serial` was already the last user of `ws`; records it as the last user either way
bool claim_workspace(const void* ws, uint64_t serial) {
    std::lock_guard<std::mutex> lock(g_ws_mu);
    auto it = g_ws_owner.find(ws);
    if (it != g_ws_owner.end()) {
        const bool same = it->second == serial;
        it->second = serial;
        return same;
    }
    if (g_ws_owner.size() >= kWsOwnerCap) g_ws_owner.clear();
    g_ws_owner.emplace(ws, serial);
    return false;
}

// Status words of runs whose work list travels as kernel parameters: such a run touches no workspace, and a plan allocates no
// device memory, so they are part of the library's device image, one for each of up to kOwnHeaders plans alive (others upload
// their lists).  Tags (report()) go on rising from one owner of a word to the next, which tells a late report of the last
// owner apart.
constexpr int kOwnHeaders = 256, kMaxDevices = 64;
__device__ WsHeader g_own_hdr[kOwnHeaders];
std::mutex g_own_mu;
int32_t g_own_given_back[kOwnHeaders], g_own_n_given_back = 0, g_own_never_used = 0;
uint32_t g_own_runs[kOwnHeaders];

int32_t acquire_own_header(uint32_t* runs) {
    std::lock_guard<std::mutex> lock(g_own_mu);
    int32_t k = -1;
    if (g_own_n_given_back > 0) k = g_own_given_back[--g_own_n_given_back];
    else if (g_own_never_used < kOwnHeaders) k = g_own_never_used++;
    if (k >= 0) *runs = g_own_runs[k];
    return k;
}

void release_own_header(int32_t k, uint32_t runs) {
    if (k < 0) return;
    std::lock_guard<std::mutex> lock(g_own_mu);
    g_own_runs[k] = runs;
    g_own_given_back[g_own_n_given_back++] = k;
}

// its address on the current device, or null
WsHeader* own_header(int32_t k) {
    static std::atomic<WsHeader*> base[kMaxDevices];
    int dev = -1;
    if (k < 0 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    WsHeader* p = base[dev].load(std::memory_order_relaxed);
    if (!p) {
        if (cudaGetSymbolAddress((void**)&p, g_own_hdr) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        base[dev].store(p, std::memory_order_relaxed);
    }
    return p + k;
}

void forget_plan(uint64_t serial) {
    std::lock_guard<std::mutex> lock(g_ws_mu);
    for (auto it = g_ws_owner.begin(); it != g_ws_owner.end();)
        it = it->second == serial ? g_ws_owner.erase(it) : std::next(it);
}

}  // namespace

struct ps_plan {
    ps_shape shape{};
    int32_t n = 0, max_pages = 0, num_sms = 0, device_sms = 0;
    // SMs given to each kernel: all of them when only one class of rows is present; in a mixed batch the
    // decode kernel (HBM-bound: a fraction of the SMs saturates the memory system) and the prefill kernel
    // (tensor-bound) run side by side on disjoint sets of SMs
    int32_t dec_sms = 0, pf_sms = 0;
    bool pairs = false;      // prefill items go to CTA pairs
    int32_t pf_workers = 0;  // what they are handed to: CTAs, or CTA pairs (one SM each)
    bool concurrent = false;
    bool decode_last = false;    // side by side, the decode kernel is predicted to end well after the prefill kernel
    bool cut_by_choice = false;  // prefill items are cut that a lean plan might leave whole
    bool tiny_as_rows = false;  // this batch runs its chunks of a few tokens as decode rows
    std::vector<DecodePiece> pieces;
    std::vector<DecodeUnit> units;
    bool cta_pieces = false;             // a CTA per piece, no units
    int dec_pages = 1;                   // pages a stage of the decode kernel with a unit per warp
    std::vector<PrefillItem> prefill;
    std::vector<MergeEntry> merge;       // prefill q tile pairs cut into segments: combined by the merge kernel
    std::vector<DecodeMerge> dmerge;     // combined inside the decode kernel
    int64_t decode_merge_rows = 0;
    std::vector<int32_t> prefill_cta_start;  // static partition: CTA b runs items [start[b], start[b+1]); empty = dynamic queue
    std::vector<int32_t> prior;  // kept for item inspection
    ps_plan_info info{};
    // workspace layout: two image slots of slot_stride bytes each, then the partial rows.  The stride only ever
    // grows (with headroom), so that re-planning to another batch normally leaves the slots and the partial
    // buffers where the runs still in flight expect them.
    size_t off_pieces = 0, off_units = 0, off_prefill = 0, off_merge = 0, off_cta_start = 0, off_dmerge = 0, off_dmerge_cnt = 0, image_bytes = 0;
    size_t slot_stride = 0;
    size_t off_part_lse = 0, off_part_o = 0, ws_bytes = 0;
    bool layout_moved = false;  // slot_stride grew since the last run: the slots of earlier runs lie elsewhere
    uint64_t serial = 0;        // identifies this plan object among all that may share a workspace
    int64_t wait_limit_ns = kDefaultWaitLimitNs;  // bound of every device-side wait of this plan's kernels
    // pinned staging image of [0, image_bytes)
    char* pinned = nullptr;
    bool pinned_is_cuda = false;
    size_t pinned_cap = 0;
    // The work-list image is uploaded on a private stream into one of two slots at the head of the
    // workspace, so that the upload for run i+1 overlaps the kernels of run i.
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_copied[2] = {nullptr, nullptr};  // slot's upload finished (copy stream)
    cudaEvent_t ev_done[2] = {nullptr, nullptr};    // the run that used the slot finished (caller's stream)
    cudaEvent_t ev_fence = nullptr;                  // caller's stream position, when the workspace changed
    cudaStream_t side_stream = nullptr;              // decode kernel of a mixed batch (runs beside the prefill kernel)
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    bool done_valid[2] = {false, false};
    bool copy_pending = false;
    int last_slot = 0;
    unsigned run_no = 0;
    void* last_ws = nullptr;
    WsHeader* last_hdr = nullptr;
    int32_t last_tag = 0;
    // Small batches: the work list travels as kernel parameters, and the run's status word is one of the library's.
    bool inline_list = false;
    int32_t own_hdr = -1;
    uint32_t inline_runs = 0;
    // optional per-kernel timing: 6 events per recorded run (begin/end of prefill, decode, merge)
    bool timing = false;
    std::vector<cudaEvent_t> tev;
    int timed_runs = 0;
};

static int query_num_sms() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

// Batches too small for a share per warp: a CTA per piece.  Applies where every (row, kv head) gets a CTA of its own and no
// piece is longer than kCtaMaxPiece -- where a warp's share would be the smallest unit, and a piece per
// warp would be many partial rows.  Rows longer than kCtaMinPiece are cut as far as there are CTAs.
static bool plan_decode_ctas(ps_plan* pl, const int32_t* prior, const int32_t* q_len, const std::vector<int32_t>& q_start, int64_t total_pages,
                             int64_t longest, int64_t* n_slots) {
    const int Hkv = pl->shape.n_kv_heads, G = pl->shape.n_q_heads / Hkv;
    const int64_t max_piece = kCtaMaxPiece;
    if (total_pages > pl->dec_sms * max_piece) return false;
    std::vector<std::pair<int32_t, int32_t>> rows;  // (request, keys the row sees)
    for (int r = 0; r < pl->n; ++r) {
        if (!runs_as_decode(pl->shape, pl->tiny_as_rows, prior[r], q_len[r])) continue;
        if ((int64_t)(rows.size() + q_len[r]) * Hkv > pl->dec_sms) return false;
        for (int i = 0; i < q_len[r]; ++i) rows.emplace_back(r, prior[r] + i + 1);
    }
    auto pages_of = [](int32_t keys) { return (int64_t)(keys + kPage - 1) / kPage; };
    auto pieces_at = [&](int64_t piece) {
        int64_t n = 0;
        for (const auto& row : rows) n += (pages_of(row.second) + piece - 1) / piece;
        return n * Hkv;
    };
    // Uncut if that leaves no warp too many pages (a list without merges need not be uploaded); else the smallest piece that
    // leaves no more pieces than CTAs.
    int64_t lo = std::max<int64_t>(kCtaMinPiece, longest <= max_piece ? longest : 0), hi = std::max(lo, longest);
    while (lo < hi) {
        const int64_t mid = (lo + hi) / 2;
        if (pieces_at(mid) <= pl->dec_sms) hi = mid; else lo = mid + 1;
    }
    if (lo > max_piece) return false;
    pl->cta_pieces = true;
    pl->info.decode_segment_tokens = (int32_t)(lo * kPage);
    pl->pieces.clear();
    pl->units.clear();
    pl->dmerge.clear();
    int32_t tok_req = -1, tok = 0;
    for (const auto& row : rows) {
        tok = row.first == tok_req ? tok + 1 : q_start[row.first];
        tok_req = row.first;
        const int64_t pages = pages_of(row.second), n_seg = (pages + lo - 1) / lo;
        for (int g = 0; g < Hkv; ++g) {
            for (int64_t s = 0; s < n_seg; ++s) {
                DecodePiece pc{};
                pc.req = row.first;
                pc.kv_head = g;
                pc.page_begin = (int32_t)(pages * s / n_seg);
                pc.page_end = (int32_t)(pages * (s + 1) / n_seg);
                pc.q_tok = tok;
                pc.part_slot = n_seg > 1 ? (int32_t)(*n_slots + s * G) : -1;
                pc.kv_len = row.second;
                pc.merge_idx = n_seg > 1 ? (int32_t)pl->dmerge.size() : 0;
                pl->pieces.push_back(pc);
            }
            if (n_seg > 1) {
                pl->dmerge.push_back(DecodeMerge{(int32_t)*n_slots, (int32_t)n_seg});
                *n_slots += n_seg * G;
            }
        }
    }
    pl->decode_merge_rows += (int64_t)pl->dmerge.size() * G;
    return true;
}

// Which form of the decode kernel with a unit per warp takes a batch at head dimension 64: two pages a stage on 12 warps an SM, or one
// on 24.  A row costs a warp some 2 us beside its pages, so short rows of which a warp has several are done sooner by twice the warps:
// from 1.2 (row, kv head)s a warp up to 5 pages a row, from 1.5 up to 9, from 2 up to 15, where the smallest units do not leave warps idle
// anyway.
// Measured (12 warps / 24, us, 8 kv heads, 1 and 4 q heads each, contexts within half of the mean): 512 rows of 28 tokens 20.5 / 18.6,
// of 40 22.6 / 19.3, of 64 26.1 / 24.3, of 96 30.0 / 30.7, of 128 35.9 / 34.7, of 190 46.6 / 45.0, of 240 52.9 / 51.8, of 256 55.5 / 55.3; 700
// of 210 62.6 / 61.2, of 240 67.9 / 68.5; 350 of 40 19.5 / 18.3, of 64 21.8 / 20.1, of 96 25.2 / 23.6, of 128 28.7 / 28.0, of 192 35.3 /
// 35.2; 280 of 64 20.3 / 18.6, of 96 21.3 / 22.4, of 192 30.7 / 31.8; 230 of 64 18.5 / 18.4, of 128 21.4 / 22.1; few pages: 512 of 20
// 16.0 / 16.4, 350 of 28 15.8 / 18.2; 2 kv heads: 512 of 128 18.7 / 19.5.
static bool one_page_a_stage(const ps_plan& pl, int64_t n_rows, int64_t total_pages) {
    const int64_t warps = (int64_t)pl.dec_sms * decode_unit_warps(64, 2);
    if (total_pages <= kDecodeMinPagesLo * warps) return false;
    // (twice the warps leave twice the partial rows, two a unit and q head at most: not where the built-in scratch might no longer do)
    const int64_t units = 2 * warps, G = pl.shape.n_q_heads / pl.shape.n_kv_heads;
    if (2 * units * G * 65 * 4 + 3 * (n_rows + 2 * units) * (int64_t)sizeof(DecodePiece) > PS_STATIC_WORKSPACE_BYTES) return false;
    return (n_rows * 5 >= warps * 6 && total_pages <= 5 * n_rows) || (n_rows * 2 >= warps * 3 && total_pages <= 9 * n_rows) ||
           (n_rows >= warps * 2 && total_pages <= 15 * n_rows);
}

static void plan_decode(ps_plan* pl, const int32_t* prior, const int32_t* q_len, const std::vector<int32_t>& q_start,
                        const ps_plan_opts* opts, bool lean, int64_t* n_slots) {
    const int Hkv = pl->shape.n_kv_heads, G = pl->shape.n_q_heads / Hkv;
    int64_t total_pages = 0, longest = 0, n_rows = 0;  // (n_rows, total_pages: of all kv heads)
    for (int r = 0; r < pl->n; ++r)
        if (runs_as_decode(pl->shape, pl->tiny_as_rows, prior[r], q_len[r]))
            for (int i = 0; i < q_len[r]; ++i, n_rows += Hkv) {
                const int64_t pages = (prior[r] + i + 1 + kPage - 1) / kPage;
                total_pages += pages * Hkv;
                longest = std::max(longest, pages);
            }
    if (total_pages == 0) {
        pl->pieces.clear();
        pl->units.clear();
        pl->dmerge.clear();
        return;
    }
    pl->cta_pieces = false;
    pl->info.decode_segment_tokens = 0;
    if (!(opts && opts->decode_segment_tokens > 0) && plan_decode_ctas(pl, prior, q_len, q_start, total_pages, longest, n_slots)) return;
    pl->dec_pages = pl->shape.head_dim == 64 && (lean || !one_page_a_stage(*pl, n_rows, total_pages)) ? 2 : 1;
    const int64_t min_pages = std::min<int64_t>(kDecodeMinPagesHi, std::max<int64_t>(kDecodeMinPagesLo, (longest + kDecodePiecesPerRow - 1) / kDecodePiecesPerRow));
    int64_t per_unit;
    if (opts && opts->decode_segment_tokens > 0) {
        per_unit = std::max(1, opts->decode_segment_tokens / kPage);
    } else {
        const int64_t target = (int64_t)pl->dec_sms * decode_unit_warps(pl->shape.head_dim, pl->dec_pages) * kDecodeUnitsPerWarp;
        per_unit = std::max<int64_t>(min_pages, (total_pages + target - 1) / target);
        // With two pages a stage a unit's last stage should be full, but not at the price of a tenth of its pages more: 30 rows of 500 tokens,
        // 8 kv heads, with 6 pages instead of 5 19.1 us, 16.9; of 900, 10 instead of 9, 20.5, 18.7; 80 of 500, 12 instead of 11, 21.1, 22.2.
        if (pl->dec_pages == 2 && (lean || per_unit > 10)) per_unit += per_unit & 1;
    }
    pl->info.decode_segment_tokens = (int32_t)(per_unit * kPage);

    // Upper bounds on the counts (a piece ends where its row or its unit ends), so that the lists are filled
    // in place and trimmed once.
    const size_t max_units = (size_t)((total_pages + per_unit - 1) / per_unit);
    pl->pieces.resize((size_t)n_rows + max_units);
    pl->units.resize(max_units);
    pl->dmerge.resize(std::min<size_t>((size_t)n_rows, max_units));
    DecodePiece* const pieces = pl->pieces.data();
    DecodeUnit* const units = pl->units.data();
    DecodeMerge* const dmerge = pl->dmerge.data();
    int32_t n_pieces = 0, n_units = 0, n_dmerge = 0;
    int64_t slots = *n_slots;
    int64_t room = 0;  // pages the open unit can still take
    for (int r = 0; r < pl->n; ++r) {
        if (!runs_as_decode(pl->shape, pl->tiny_as_rows, prior[r], q_len[r])) continue;
        for (int i = 0; i < q_len[r]; ++i) {  // one row per new token (a decode request has one)
            const int kv_len = prior[r] + i + 1;
            const int pages = (kv_len + kPage - 1) / kPage;
            const int32_t q_tok = q_start[r] + i;
            for (int g = 0; g < Hkv; ++g) {
                const int32_t first_piece = n_pieces;
                int pg = 0;
                while (pg < pages) {
                    if (room == 0) {
                        if (n_units > 0) units[n_units - 1].piece_end = n_pieces;
                        units[n_units++].piece_begin = n_pieces;
                        room = per_unit;
                    }
                    const int take = (int)std::min<int64_t>(room, pages - pg);
                    DecodePiece& pc = pieces[n_pieces++];
                    pc.req = r;
                    pc.kv_head = g;
                    pc.page_begin = pg;
                    pc.page_end = pg + take;
                    pc.q_tok = q_tok;
                    pc.part_slot = -1;
                    pc.kv_len = kv_len;
                    pc.merge_idx = 0;
                    pg += take;
                    room -= take;
                }
                const int32_t cnt = n_pieces - first_piece;
                if (cnt > 1) {
                    for (int32_t s = 0; s < cnt; ++s) {
                        pieces[first_piece + s].part_slot = (int32_t)(slots + (int64_t)s * G);
                        pieces[first_piece + s].merge_idx = n_dmerge;
                    }
                    dmerge[n_dmerge].base = (int32_t)slots;
                    dmerge[n_dmerge].n_seg = cnt;
                    ++n_dmerge;
                    slots += (int64_t)cnt * G;
                }
            }
        }
    }
    if (n_units > 0) units[n_units - 1].piece_end = n_pieces;
    pl->pieces.resize((size_t)n_pieces);
    pl->units.resize((size_t)n_units);
    pl->dmerge.resize((size_t)n_dmerge);
    pl->decode_merge_rows += (int64_t)n_dmerge * G;
    *n_slots = slots;
}

constexpr double kPrefillWholeItemSlack = 1.12;  // uncut items are taken if the busiest CTA stays within this of an even split
constexpr double kPrefillMinCtaCost = 4.0;  // do not spread the work thinner than this per CTA (two key tiles)

static void plan_prefill(ps_plan* pl, const int32_t* prior, const int32_t* q_len, const std::vector<int32_t>& q_start,
                         const ps_plan_opts* opts, bool lean, int64_t* n_slots) {
    const int Hkv = pl->shape.n_kv_heads, G = pl->shape.n_q_heads / Hkv;
    const int tile_tok = kPrefillRowsPerItem / G;
    const PrefillModel usual = prefill_model(pl->shape, pl->pairs), lean_cost = lean_model(pl->shape, usual), &cost = lean ? lean_cost : usual;
    pl->cut_by_choice = false;
    struct Tile { int r, g, tok0, n_tok, first_pos, key_tiles; };
    std::vector<Tile> tiles;
    size_t n_tiles = 0;
    for (int r = 0; r < pl->n; ++r)
        if (!runs_as_decode(pl->shape, pl->tiny_as_rows, prior[r], q_len[r])) n_tiles += (size_t)((q_len[r] + tile_tok - 1) / tile_tok) * Hkv;
    tiles.reserve(n_tiles);
    int64_t total_key_tiles = 0;
    for (int r = 0; r < pl->n; ++r) {
        if (runs_as_decode(pl->shape, pl->tiny_as_rows, prior[r], q_len[r])) continue;
        for (int g = 0; g < Hkv; ++g)
            for (int t0 = 0; t0 < q_len[r]; t0 += tile_tok) {
                const int n_tok = std::min(tile_tok, q_len[r] - t0);
                const int first_pos = prior[r] + t0;
                const int kt = (first_pos + n_tok + kPrefillKeyTile - 1) / kPrefillKeyTile;
                tiles.push_back(Tile{r, g, t0, n_tok, first_pos, kt});
                total_key_tiles += kt;
            }
    }
    pl->prefill_cta_start.clear();
    if (tiles.empty()) return;
    const bool many_short = pl->shape.head_dim == 128 && !pl->pairs;  // (cutting them never pays)

    // (tile, key-tile index) of every cut, ascending in both: tile i is cut into pieces at these key tiles
    // (exclusive of 0 and key_tiles)
    struct Cut { int tile, at; };
    std::vector<Cut> cuts;
    // owner CTA of the first piece of each tile and of each following piece, for the static partition
    bool static_partition = false, whole_items = false;
    if (opts && opts->prefill_segment_tokens > 0) {
        const int seg_tiles = std::max(1, opts->prefill_segment_tokens / kPrefillKeyTile);
        pl->info.prefill_segment_tokens = seg_tiles * kPrefillKeyTile;
        for (size_t i = 0; i < tiles.size(); ++i) {
            const int n_seg = (tiles[i].key_tiles + seg_tiles - 1) / seg_tiles;
            const int base_tiles = tiles[i].key_tiles / n_seg, extra = tiles[i].key_tiles % n_seg;
            int kt0 = 0;
            for (int s = 0; s + 1 < n_seg; ++s) {
                kt0 += base_tiles + (s < extra ? 1 : 0);
                cuts.push_back(Cut{(int)i, kt0});
            }
        }
    } else if ((int64_t)tiles.size() < 4LL * pl->num_sms && !many_short) {
        // Few items per SM of all the device has, whatever the prefill kernel's share: the shares are planned to end together,
        // and then the helpers that a queue brings find it empty 6 us behind the decode kernel's end (128 rows of about 2500
        // tokens and 256 items on 60 SMs 224 us, 236 from a queue).  Give every CTA an equal share of the flattened (item, key
        // tile) cost line, cutting items where a share ends.  Only the cut items need the merge.
        static_partition = true;
        double total = 0;
        for (const Tile& t : tiles) total += cost.fixed + t.key_tiles + cost.masked_extra;
        // (No two items on one CTA while another has none: two fresh items of one key tile, 16 q / 2 kv heads of 64, 14.1 us on one
        // CTA, 9.7 on two; 56 items of 1 and 2 key tiles 15.2 on 50 CTAs, 12.0 on 56.)
        const int n_cta = (int)std::max<double>(1, std::min<double>(pl->pf_workers, std::max<double>(lean ? 0 : (double)tiles.size(), total / kPrefillMinCtaCost)));
        // Many short items (fresh prompts): whole items, longest first, each to the CTA with the least work so far.
        // If that comes within kPrefillWholeItemSlack of an even split, nothing is cut: no partial rows, no merge
        // kernel, no item paying its fixed cost twice.
        {
            std::vector<int> order(tiles.size());
            for (size_t i = 0; i < tiles.size(); ++i) order[i] = (int)i;
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return tiles[a].key_tiles > tiles[b].key_tiles; });
            // (least work so far, CTA): equal loads go to the lower CTA
            typedef std::pair<double, int> Slot;
            std::vector<Slot> heap((size_t)n_cta);
            for (int c = 0; c < n_cta; ++c) heap[c] = Slot(0.0, c);  // ascending: already a min-heap under greater<>
            std::vector<int> owner(tiles.size());
            std::vector<int32_t> count((size_t)n_cta + 1, 0);
            double makespan = 0;
            for (int i : order) {
                std::pop_heap(heap.begin(), heap.end(), std::greater<Slot>());
                Slot& least = heap.back();
                owner[i] = least.second;
                ++count[least.second + 1];
                least.first += cost.fixed + tiles[i].key_tiles + cost.masked_extra;
                makespan = std::max(makespan, least.first);
                std::push_heap(heap.begin(), heap.end(), std::greater<Slot>());
            }
            const double whole = (int64_t)tiles.size() <= kFewItems ? cost.whole_few : cost.whole;
            // (cutting is not free either, and from four items a worker on it has less to gain than the partial rows cost in
            // space, 19 MB in a batch that needs none)
            if ((int64_t)tiles.size() >= 4LL * pl->pf_workers || makespan <= std::max(kPrefillWholeItemSlack * total / n_cta, total / n_cta + whole)) {
                for (int c = 0; c < n_cta; ++c) count[c + 1] += count[c];
                pl->prefill_cta_start.assign(count.begin(), count.end());
                std::vector<Tile> sorted(tiles.size());
                for (int i : order) sorted[(size_t)count[owner[i]]++] = tiles[i];  // each CTA's items longest first
                tiles.swap(sorted);
                whole_items = true;
            } else {
                pl->cut_by_choice = makespan <= total / n_cta + lean_cost.whole + 1 || (int64_t)tiles.size() * 4 >= 15LL * pl->pf_workers;
            }
        }
        if (!whole_items) {
        // CTA k ends where the running cost passes (k + 1) * quota (absolute marks, so rounding does not pile
        // up).  A share that ends inside an item makes the rest of that item pay the fixed cost again, and how
        // many shares do depends on the quota itself: bisect for the smallest quota that does not leave the
        // last CTA with more than a share.
        int n_items = 0;
        double q_lo = total / n_cta, q_hi = (total + (n_cta - 1) * cost.fixed) / n_cta + 0.5;
        for (int pass = 0; pass < 7; ++pass) {
            const double quota = pass == 6 ? q_hi : 0.5 * (q_lo + q_hi);  // the last pass keeps a quota known to fit
            pl->prefill_cta_start.assign(1, 0);
            cuts.clear();
            n_items = 0;
            int cta = 0;
            double cum = 0, cum_at_last = 0;  // cost handed out so far; and before the last CTA
            auto close_cta = [&]() {
                ++cta;
                pl->prefill_cta_start.push_back(n_items);
                if (cta == n_cta - 1) cum_at_last = cum;
            };
            for (size_t i = 0; i < tiles.size(); ++i) {
                const int kt = tiles[i].key_tiles;
                int kt0 = 0;
                for (;;) {
                    const double rest = cost.fixed + (kt - kt0) + cost.masked_extra;  // the item's remaining tiles as one piece
                    const double room = (cta + 1) * quota - cum;
                    const bool cta_has_work = pl->prefill_cta_start.back() < n_items;
                    const double fit = room - cost.fixed;
                    const int take = fit < 0.5 ? 0 : (int)(fit + 0.5);  // key tiles that fit, to the nearest
                    if (cta == n_cta - 1 || rest <= room + 0.5 || take >= kt - kt0 || (take < 1 && !cta_has_work)) {
                        cum += rest;
                        ++n_items;
                        break;
                    }
                    if (take >= 1) {
                        kt0 += take;
                        cuts.push_back(Cut{(int)i, kt0});
                        cum += cost.fixed + take;
                        ++n_items;
                    }
                    close_cta();  // (with take < 1: no room left for even one key tile; the item starts in the next CTA)
                }
                while (cta < n_cta - 1 && cum >= (cta + 1) * quota - 0.5) close_cta();
            }
            const bool fits = cta < n_cta - 1 || cum - cum_at_last <= quota + 0.5;
            if (fits) q_hi = quota; else q_lo = quota;
        }
        while ((int)pl->prefill_cta_start.size() < n_cta) pl->prefill_cta_start.push_back(n_items);  // CTAs left without work
        pl->prefill_cta_start.push_back(n_items);
        }
    }

    pl->prefill.reserve(tiles.size() + cuts.size());
    size_t next_cut = 0;
    for (size_t i = 0; i < tiles.size(); ++i) {
        const Tile& t = tiles[i];
        const size_t first_cut = next_cut;
        while (next_cut < cuts.size() && cuts[next_cut].tile == (int)i) ++next_cut;
        const int n_seg = (int)(next_cut - first_cut) + 1;
        const int visible = t.first_pos + t.n_tok;
        int32_t slot_base = -1;
        if (n_seg > 1) {
            slot_base = (int32_t)*n_slots;
            MergeEntry me{};
            me.q_tok = q_start[t.r] + t.tok0;
            me.n_tok = t.n_tok;
            me.kv_head = t.g;
            me.base = slot_base;
            me.n_seg = n_seg;
            me.seg_stride = t.n_tok * G;
            pl->merge.push_back(me);
            *n_slots += (int64_t)n_seg * t.n_tok * G;
        }
        for (int s = 0; s < n_seg; ++s) {
            const int kt0 = s == 0 ? 0 : cuts[first_cut + s - 1].at;
            const int kt1 = s == n_seg - 1 ? t.key_tiles : cuts[first_cut + s].at;
            PrefillItem it{};
            it.req = t.r;
            it.kv_head = t.g;
            it.key_begin = kt0 * kPrefillKeyTile;
            it.key_end = std::min(visible, kt1 * kPrefillKeyTile);
            it.q_tok = q_start[t.r] + t.tok0;
            it.n_tok = t.n_tok;
            it.part_slot = n_seg > 1 ? slot_base + s * t.n_tok * G : -1;
            it.first_pos = t.first_pos;
            pl->prefill.push_back(it);
        }
    }
    if (!static_partition) {
        // dynamic queue: longest first, so that it finishes with the short items
        std::stable_sort(pl->prefill.begin(), pl->prefill.end(), [](const PrefillItem& a, const PrefillItem& b) {
            return (a.key_end - a.key_begin) > (b.key_end - b.key_begin);
        });
    }
}

extern "C" {

ps_status ps_attn_plan(const ps_shape* shape, const int32_t* prior_host, const int32_t* q_len_host, int32_t n,
                       int32_t max_pages_per_seq, const ps_plan_opts* opts, ps_plan** plan_inout,
                       size_t* workspace_bytes_out) {
    ps_status st = check_shape(shape);
    if (st != PS_OK) return st;
    if (!prior_host || !q_len_host || !plan_inout || !workspace_bytes_out) return fail(PS_ERR_INVALID, "null argument");
    if (n < 1) return fail(PS_ERR_INVALID, "n=%d must be positive", n);
    if (max_pages_per_seq < 1) return fail(PS_ERR_INVALID, "max_pages_per_seq=%d must be positive", max_pages_per_seq);
    if (opts && (opts->decode_segment_tokens < 0 || opts->decode_segment_tokens % kPage != 0))
        return fail(PS_ERR_INVALID, "decode_segment_tokens must be a non-negative multiple of %d", kPage);
    if (opts && (opts->prefill_segment_tokens < 0 || opts->prefill_segment_tokens % kPrefillKeyTile != 0))
        return fail(PS_ERR_INVALID, "prefill_segment_tokens must be a non-negative multiple of %d", kPrefillKeyTile);
    std::vector<int32_t> q_start((size_t)n + 1);
    int64_t T = 0;
    for (int r = 0; r < n; ++r) {
        if (q_len_host[r] < 1) return fail(PS_ERR_INVALID, "request %d: q_len=%d must be >= 1", r, q_len_host[r]);
        if (prior_host[r] < 0) return fail(PS_ERR_INVALID, "request %d: prior=%d must be >= 0", r, prior_host[r]);
        if ((int64_t)prior_host[r] + q_len_host[r] > (int64_t)max_pages_per_seq * kPage)
            return fail(PS_ERR_INVALID, "request %d: kv_len=%lld exceeds max_pages_per_seq * page_size", r,
                        (long long)prior_host[r] + q_len_host[r]);
        if (shape->dtype == 1 && q_len_host[r] != 1)
            return fail(PS_ERR_UNSUPPORTED, "request %d: q_len=%d -- the FP8 cache variant serves decode rows (q_len = 1) only", r,
                        q_len_host[r]);
        q_start[r] = (int32_t)T;
        T += q_len_host[r];
        if (T > (1 << 24)) return fail(PS_ERR_INVALID, "more than 2^24 new tokens in one batch");
    }
    q_start[n] = (int32_t)T;

    ps_plan* pl = *plan_inout;
    const bool fresh = pl == nullptr;
    if (fresh) {
        pl = new (std::nothrow) ps_plan();
        if (!pl) return fail(PS_ERR_OOM, "host allocation failed");
        pl->serial = next_plan_serial();
        pl->own_hdr = acquire_own_header(&pl->inline_runs);
    } else if (pl->copy_pending && pl->ev_copied[pl->last_slot]) {
        cudaError_t e = cudaEventSynchronize(pl->ev_copied[pl->last_slot]);
        if (e != cudaSuccess) return fail(PS_ERR_CUDA, "cudaEventSynchronize failed: %s", cudaGetErrorString(e));
        pl->copy_pending = false;
    }
    pl->shape = *shape;
    pl->n = n;
    pl->max_pages = max_pages_per_seq;
    if (opts && opts->num_sms > 0) {
        pl->num_sms = opts->num_sms;
    } else {
        if (pl->device_sms <= 0) pl->device_sms = query_num_sms();
        pl->num_sms = pl->device_sms;
    }
    if (pl->num_sms <= 0) {
        if (fresh) ps_plan_free(pl);
        return fail(PS_ERR_CUDA, "no CUDA device to plan for (pass opts->num_sms to plan without one)");
    }
    pl->prefill.clear();
    pl->merge.clear();
    pl->decode_merge_rows = 0;
    pl->prior.assign(prior_host, prior_host + n);
    pl->info = ps_plan_info{};
    {
        double true_dec_bytes = 0;
        for (int r = 0; r < n; ++r)
            if (q_len_host[r] == 1) true_dec_bytes += ((double)prior_host[r] + 1.0) * 2.0 * shape->n_kv_heads * shape->head_dim * 2.0;
        // (forced prefill segments: the caller wants every chunk on the prefill kernel)
        pl->tiny_as_rows = !(opts && opts->prefill_segment_tokens > 0) && true_dec_bytes <= kTinyChunkMaxDecodeBytes;
    }
    {
        const int tile_tok = kPrefillRowsPerItem / (shape->n_q_heads / shape->n_kv_heads);
        int64_t items = 0, key_tiles = 0;
        for (int r = 0; r < n; ++r) {
            if (runs_as_decode(*shape, pl->tiny_as_rows, prior_host[r], q_len_host[r])) continue;
            for (int t0 = 0; t0 < q_len_host[r]; t0 += tile_tok) {
                items += shape->n_kv_heads;
                key_tiles += (int64_t)shape->n_kv_heads * ((prior_host[r] + std::min(t0 + tile_tok, q_len_host[r]) + kPrefillKeyTile - 1) / kPrefillKeyTile);
            }
        }
        // (forced segments: the kernel of the larger batches)
        pl->pairs = (opts && opts->prefill_segment_tokens > 0) ? shape->head_dim == 128 : prefill_on_pairs(*shape, pl->num_sms, items, key_tiles);
    }
    // ---- split the SMs between the two kernels of a mixed batch ----
    {
        double longest = 0;                  // steps of the longest prefill item
        double dec_bytes = 0, pf_steps = 0;  // KV bytes the decode rows stream; key-tile steps of the prefill items
        double dec_rows = 0;                 // (row, kv head)s
        const int G = shape->n_q_heads / shape->n_kv_heads;
        const PrefillModel cost = measured_model(pl->shape, prefill_model(pl->shape, pl->pairs));
        const int tile_tok = kPrefillRowsPerItem / G;
        for (int r = 0; r < n; ++r) {
            if (runs_as_decode(*shape, pl->tiny_as_rows, prior_host[r], q_len_host[r])) {
                dec_rows += (double)q_len_host[r] * shape->n_kv_heads;
                for (int i = 0; i < q_len_host[r]; ++i)
                    dec_bytes += ((double)prior_host[r] + i + 1.0) * 2.0 * shape->n_kv_heads * shape->head_dim * 2.0;
            } else {
                for (int t0 = 0; t0 < q_len_host[r]; t0 += tile_tok) {
                    const int n_tok = std::min(tile_tok, q_len_host[r] - t0);
                    const double steps = cost.fixed + (prior_host[r] + t0 + n_tok + kPrefillKeyTile - 1) / kPrefillKeyTile;
                    pf_steps += steps * shape->n_kv_heads;
                    longest = std::max(longest, steps);
                }
            }
        }
        pl->dec_sms = pl->pf_sms = pl->num_sms;
        pl->concurrent = pl->decode_last = false;
        // Decode rows alone stream a little faster from 128 SMs on most GPUs: all 148 ask for more than HBM gives, and their requests get
        // in each other's way.  (A number of SMs and no share of them, because it is their requests that count; 136 and 140 are slower
        // than both.)  The time on 148 SMs over that on 128, both in turn on one GPU, 45 to 81 batches of 0.8 to 19 GB, head dimensions 64
        // and 128, even, uniform and lognormal contexts, geometric means: 1.032, 1.033, 1.036, 1.031 on four GPUs and 0.975 on a fifth; at
        // 0.8 GB 1.019 to 1.035 and 0.980, at 19 GB 1.039 to 1.049 and 0.972: no end of the range in sight.  Below the line, 0.4 and
        // 0.6 GB, 0.99 to 1.01.  Not for the FP8 cache, whose pages cost the SMs too much arithmetic.
        if (pf_steps == 0 && shape->dtype == 0 && dec_bytes >= kDecodeManyBytes) pl->dec_sms = std::min(pl->num_sms, kDecodeAloneSms);
        if (dec_bytes > 0 && pf_steps > 0 && pl->num_sms >= 16) {
            // time models (seconds): decode = bytes / min(side-by-side peak, n * per-SM rate); prefill = steps * step time / m
            auto t_dec = [&](int nd) { return dec_bytes / std::min(kDecodeSharedPeakBytesPerSec, nd * decode_rate_per_sm(*shape)) + kKernelFloorSec; };
            // Whole items leave some workers idle at the end (about 0.4 of the longest item on average) and take at least the
            // longest one; cutting them costs cost.cut steps instead.
            auto pf_time = [&](int sms) {
                const double even = pf_steps * cost.step_sec / sms, worker_step = cost.step_sec / cost.sms_per_worker;
                return std::min(std::max(even + 0.4 * longest * worker_step, longest * worker_step), even + cost.cut * worker_step);
            };
            auto t_pf = [&](int nd) { return pf_time(pl->num_sms - nd) + kKernelFloorSec; };
            int best_n = 0;
            double best_t = 1e30;
            for (int nd = 8; nd <= pl->num_sms - 8; nd += 4) {
                const double t = std::max(t_dec(nd), t_pf(nd));
                if (t < best_t) {
                    best_t = t;
                    best_n = nd;
                }
            }
            // Once the decode rows saturate HBM the modelled time is flat in n; measured step times keep
            // improving a little as the decode kernel gets more SMs, as long as the prefill kernel still ends
            // well before it.  Take the middle of that flat stretch.  (Not at head dimension 64, where it begins at some 84 SMs and
            // more of them gain nothing: from its beginning / its middle 400 rows of about 1000 tokens and a fresh 1024-token chunk
            // 133 / 140 us, on 2000 141 / 140, 256 of 2000 and 512 on 1000 166 / 176, 100 of 4000 and 700 on 500 129 / 137.)
            int hi = best_n;
            for (int nd = best_n; shape->head_dim == 128 && nd <= pl->num_sms - 8; nd += 4)
                if (std::max(t_dec(nd), t_pf(nd)) <= 1.015 * best_t && t_pf(nd) <= 0.8 * t_dec(nd)) hi = nd;
            best_n = (best_n + hi) / 2 / 4 * 4;
            const double t_seq = dec_bytes / kDecodePeakBytesPerSec + pf_time(pl->num_sms) + 2 * kKernelFloorSec;
            // The decode rows pay the shared rate only while the prefill kernel runs; once it has ended they stream
            // at the rate their CTAs reach alone.  A short chunk beside many decode rows is therefore cheaper than
            // the model above says, which matters for the choice against running the two one after the other.
            if (best_n > 0) {
                const double pf_work = pf_time(pl->num_sms - best_n);
                const double shared = std::min(kDecodeSharedPeakBytesPerSec, best_n * decode_rate_per_sm(*shape));
                const double alone = std::min(kDecodePeakBytesPerSec, best_n * decode_alone_rate_per_sm(*shape));
                const double dec_work = dec_bytes <= shared * pf_work ? dec_bytes / shared : pf_work + (dec_bytes - shared * pf_work) / alone;
                best_t = std::min(best_t, std::max(pf_work, dec_work) + kKernelFloorSec);
            }
            if (best_n > 0 && best_t < 0.95 * t_seq) {
                pl->dec_sms = best_n;
                pl->pf_sms = pl->num_sms - best_n;
                pl->concurrent = true;
                const double rows_per_warp = dec_rows / (best_n * decode_unit_warps(shape->head_dim, 2));
                const double warp_sec = kRowSec * rows_per_warp + kSegmentSec * std::max(0.0, 1 / rows_per_warp - 1);
                pl->decode_last = t_dec(best_n) + warp_sec - t_pf(best_n) >= kMergeUnderDecodeSec;
            }
        }
        pl->pf_workers = std::max(1, pl->pf_sms / prefill_model(pl->shape, pl->pairs).sms_per_worker);
    }
    const int d = shape->head_dim;
    // (re)size the slots with headroom: a batch of the next iterations that needs a somewhat longer work list still fits, and the
    // layout stays put
    auto stride_for = [](size_t image_bytes) { return align_up(image_bytes + image_bytes / 2, 4096); };
    auto lay_out_image = [pl]() {
        size_t off = 256;  // WsHeader
        pl->off_pieces = off;   off = align_up(off + pl->pieces.size() * sizeof(DecodePiece), 256);
        pl->off_units = off;    off = align_up(off + pl->units.size() * sizeof(DecodeUnit), 256);
        pl->off_prefill = off;  off = align_up(off + pl->prefill.size() * sizeof(PrefillItem), 256);
        pl->off_merge = off;    off = align_up(off + pl->merge.size() * sizeof(MergeEntry), 256);
        pl->off_dmerge = off;   off = align_up(off + pl->dmerge.size() * sizeof(DecodeMerge), 256);
        pl->off_dmerge_cnt = off; off = align_up(off + pl->dmerge.size() * sizeof(int32_t), 256);
        pl->off_cta_start = off; off = align_up(off + pl->prefill_cta_start.size() * sizeof(int32_t), 256);
        pl->image_bytes = off;
    };
    int64_t n_slots = 0;
    auto plan_items = [&](bool lean) {
        pl->prefill.clear();
        pl->merge.clear();
        pl->decode_merge_rows = 0;
        n_slots = 0;
        plan_decode(pl, prior_host, q_len_host, q_start, opts, lean, &n_slots);
        plan_prefill(pl, prior_host, q_len_host, q_start, opts, lean, &n_slots);
        lay_out_image();
        return 2 * std::max(pl->slot_stride, pl->image_bytes > pl->slot_stride ? stride_for(pl->image_bytes) : 0) + (size_t)n_slots * (d + 1) * sizeof(float) + 512;
    };
    // Items that are cut because their merge is quick, and twice the decode warps beside cut items, leave more partial rows: where the
    // built-in scratch would no longer do because of them, the batch is planned with fewer.
    const size_t need = plan_items(false);
    const bool twice_the_warps = d == 64 && !pl->units.empty() && pl->dec_pages == 1 && !pl->merge.empty();
    if (need > PS_STATIC_WORKSPACE_BYTES && (twice_the_warps || pl->cut_by_choice || (d == 64 && need <= PS_STATIC_WORKSPACE_BYTES / 10 * 11))) plan_items(true);
    pl->inline_list = (pl->pieces.empty() || (pl->cta_pieces && pl->dmerge.empty() && pl->pieces.size() <= kInlinePieces)) &&
                      (pl->prefill.empty() || (pl->prefill.size() <= kInlineItems && pl->merge.empty() && !pl->prefill_cta_start.empty() &&
                                               pl->prefill_cta_start.size() <= kInlineStarts));
    if (n_slots > 0x7fffffffLL) {
        if (fresh) ps_plan_free(pl);
        return fail(PS_ERR_UNSUPPORTED, "partial buffer would need %lld slots", (long long)n_slots);
    }

    if (pl->image_bytes > pl->slot_stride) {
        pl->slot_stride = stride_for(pl->image_bytes);
        pl->layout_moved = true;
    }
    size_t off = 2 * pl->slot_stride;  // two image slots
    pl->off_part_lse = off; off = align_up(off + (size_t)n_slots * sizeof(float), 256);
    pl->off_part_o = off;   off = align_up(off + (size_t)n_slots * d * sizeof(float), 256);
    pl->ws_bytes = off;

    if (pl->pinned_cap < pl->image_bytes) {
        if (pl->pinned) { if (pl->pinned_is_cuda) cudaFreeHost(pl->pinned); else free(pl->pinned); }
        pl->pinned = nullptr;
        const size_t cap = std::max(pl->image_bytes * 2, (size_t)1 << 16);
        // Page-locked staging lets the work-list upload run asynchronously.  Without a CUDA
        // device (planning ahead of time on another host) plain memory holds the image.
        pl->pinned_is_cuda = cudaHostAlloc((void**)&pl->pinned, cap, cudaHostAllocDefault) == cudaSuccess;
        if (!pl->pinned_is_cuda) {
            (void)cudaGetLastError();
            pl->pinned = (char*)malloc(cap);
        }
        if (!pl->pinned) {
            pl->pinned_cap = 0;
            if (fresh) ps_plan_free(pl);
            return fail(PS_ERR_OOM, "cannot allocate %zu bytes of staging memory", cap);
        }
        pl->pinned_cap = cap;
    }
    if (!pl->copy_stream && pl->pinned_is_cuda) {
        bool ok = cudaStreamCreateWithFlags(&pl->copy_stream, cudaStreamNonBlocking) == cudaSuccess;
        for (int b = 0; b < 2 && ok; ++b)
            ok = cudaEventCreateWithFlags(&pl->ev_copied[b], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&pl->ev_done[b], cudaEventDisableTiming) == cudaSuccess;
        ok = ok && cudaEventCreateWithFlags(&pl->ev_fence, cudaEventDisableTiming) == cudaSuccess;
        ok = ok && cudaStreamCreateWithFlags(&pl->side_stream, cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&pl->ev_fork, cudaEventDisableTiming) == cudaSuccess &&
             cudaEventCreateWithFlags(&pl->ev_join, cudaEventDisableTiming) == cudaSuccess;
        if (!ok) {
            (void)cudaGetLastError();
            if (pl->copy_stream) cudaStreamDestroy(pl->copy_stream);
            pl->copy_stream = nullptr;  // uploads then go on the caller's stream
            if (pl->side_stream) cudaStreamDestroy(pl->side_stream);
            pl->side_stream = nullptr;  // mixed batches then run their two kernels one after the other
        }
    }
    memset(pl->pinned, 0, 256);
    if (!pl->pieces.empty()) memcpy(pl->pinned + pl->off_pieces, pl->pieces.data(), pl->pieces.size() * sizeof(DecodePiece));
    if (!pl->units.empty()) memcpy(pl->pinned + pl->off_units, pl->units.data(), pl->units.size() * sizeof(DecodeUnit));
    if (!pl->prefill.empty()) memcpy(pl->pinned + pl->off_prefill, pl->prefill.data(), pl->prefill.size() * sizeof(PrefillItem));
    if (!pl->merge.empty()) memcpy(pl->pinned + pl->off_merge, pl->merge.data(), pl->merge.size() * sizeof(MergeEntry));
    if (!pl->dmerge.empty()) {
        memcpy(pl->pinned + pl->off_dmerge, pl->dmerge.data(), pl->dmerge.size() * sizeof(DecodeMerge));
        memset(pl->pinned + pl->off_dmerge_cnt, 0, pl->dmerge.size() * sizeof(int32_t));  // arrival counters start at zero
    }
    if (!pl->prefill_cta_start.empty())
        memcpy(pl->pinned + pl->off_cta_start, pl->prefill_cta_start.data(), pl->prefill_cta_start.size() * sizeof(int32_t));

    pl->info.n_decode_items = (int32_t)pl->pieces.size();
    pl->info.n_prefill_items = (int32_t)pl->prefill.size();
    int64_t merge_rows = pl->decode_merge_rows;
    for (const MergeEntry& me : pl->merge) merge_rows += (int64_t)me.n_tok * (shape->n_q_heads / shape->n_kv_heads);
    pl->info.n_merge_rows = (int32_t)merge_rows;
    pl->info.n_partial_slots = n_slots;
    pl->info.total_q_tokens = T;
    pl->info.decode_sms = pl->dec_sms;
    pl->info.prefill_sms = pl->pf_sms;
    pl->info.n_launches = (pl->concurrent && !pl->pieces.empty() && pl->prefill_cta_start.empty() && (int)pl->prefill.size() > pl->pf_workers ? 1 : 0) + (pl->pieces.empty() ? 0 : 1) + (pl->prefill.empty() ? 0 : 1) + (pl->merge.empty() ? 0 : 1);
    *plan_inout = pl;
    *workspace_bytes_out = pl->ws_bytes;
    return PS_OK;
}

ps_status ps_plan_free(ps_plan* pl) {
    if (!pl) return PS_OK;
    forget_plan(pl->serial);
    if (pl->copy_stream) {
        cudaStreamSynchronize(pl->copy_stream);
        cudaStreamDestroy(pl->copy_stream);
    }
    for (int b = 0; b < 2; ++b) {
        if (pl->ev_copied[b]) cudaEventDestroy(pl->ev_copied[b]);
        if (pl->ev_done[b]) cudaEventDestroy(pl->ev_done[b]);
    }
    if (pl->ev_fence) cudaEventDestroy(pl->ev_fence);
    if (pl->side_stream) {
        cudaStreamSynchronize(pl->side_stream);
        cudaStreamDestroy(pl->side_stream);
    }
    if (pl->ev_fork) cudaEventDestroy(pl->ev_fork);
    if (pl->ev_join) cudaEventDestroy(pl->ev_join);
    for (cudaEvent_t e : pl->tev) cudaEventDestroy(e);
    release_own_header(pl->own_hdr, pl->inline_runs);
    if (pl->pinned) { if (pl->pinned_is_cuda) cudaFreeHost(pl->pinned); else free(pl->pinned); }
    delete pl;
    return PS_OK;
}

ps_status ps_plan_get_info(const ps_plan* pl, ps_plan_info* info_out) {
    if (!pl || !info_out) return fail(PS_ERR_INVALID, "null argument");
    *info_out = pl->info;
    return PS_OK;
}

ps_status ps_plan_get_items(const ps_plan* pl, int32_t* decode_items_out, int64_t decode_capacity,
                            int32_t* prefill_items_out, int64_t prefill_capacity) {
    if (!pl) return fail(PS_ERR_INVALID, "null argument");
    if (decode_items_out) {
        if (decode_capacity < (int64_t)pl->pieces.size()) return fail(PS_ERR_INVALID, "decode capacity too small");
        for (size_t i = 0; i < pl->pieces.size(); ++i) {
            const DecodePiece& pc = pl->pieces[i];
            int32_t* o = decode_items_out + 8 * i;
            o[0] = pc.req;
            o[1] = pc.kv_head;
            o[2] = pc.page_begin * kPage;
            o[3] = std::min(pc.page_end * kPage, pc.kv_len);
            o[4] = pc.q_tok;
            o[5] = 1;
            o[6] = pc.part_slot;
            o[7] = pc.kv_len - 1;  // the row's own position
        }
    }
    if (prefill_items_out) {
        if (prefill_capacity < (int64_t)pl->prefill.size()) return fail(PS_ERR_INVALID, "prefill capacity too small");
        static_assert(sizeof(PrefillItem) == 32, "item record is 8 int32");
        if (!pl->prefill.empty()) memcpy(prefill_items_out, pl->prefill.data(), pl->prefill.size() * sizeof(PrefillItem));
    }
    return PS_OK;
}

ps_status ps_attn_run(ps_plan* pl, const ps_kv* kv, const void* q_dev, const int32_t* block_table_dev, void* out_dev,
                      float* lse_out_dev, void* workspace_dev, size_t workspace_bytes, void* stream) {
    if (!pl || !kv || !q_dev || !block_table_dev || !out_dev || !workspace_dev) return fail(PS_ERR_INVALID, "null argument");
    if (workspace_bytes < pl->ws_bytes)
        return fail(PS_ERR_WORKSPACE, "workspace has %zu bytes, the plan needs %zu", workspace_bytes, pl->ws_bytes);
    if ((uintptr_t)workspace_dev % 256 != 0) return fail(PS_ERR_INVALID, "workspace must be 256-byte aligned");
    if (((uintptr_t)q_dev | (uintptr_t)out_dev) % 16 != 0) return fail(PS_ERR_INVALID, "q and out must be 16-byte aligned");
    const KvPool& pool = pool_of(kv);
    if (memcmp(&pool.shape, &pl->shape, sizeof(ps_shape)) != 0) return fail(PS_ERR_INVALID, "plan and pool shapes differ");
    cudaStream_t s = (cudaStream_t)stream;
    char* const ws_base = (char*)workspace_dev;
    const int slot = (int)(pl->run_no & 1u);
    char* ws = ws_base + (size_t)slot * pl->slot_stride;  // this run's image slot; partials are addressed from ws_base
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    PS_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    // The upload may run under the kernels of the previous run only if this plan's own record of the two slots is
    // all there is to know about the workspace: same memory as last time, slots where they were, and no other
    // plan's run on it since.
    WsHeader* const own_hdr = pl->inline_list && !capturing ? own_header(pl->own_hdr) : nullptr;  // (a graph's replays copy the staging image)
    const bool as_params = own_hdr != nullptr;
    const bool known = !as_params && claim_workspace(workspace_dev, pl->serial) && pl->last_ws == workspace_dev && !pl->layout_moved;
    if (as_params) {
        // nothing to upload, and nothing of the workspace is used
    } else if (capturing) {
        // Inside a stream capture the upload is a node of the graph on the caller's stream: every replay copies the
        // staging image as it then stands.  Nothing recorded here may be waited for by a later call outside the
        // capture, so the slot bookkeeping starts afresh.
        PS_CUDA_TRY(cudaMemcpyAsync(ws, pl->pinned, pl->image_bytes, cudaMemcpyHostToDevice, s));
        pl->done_valid[0] = pl->done_valid[1] = false;
    } else if (pl->copy_stream) {
        cudaStream_t cs = pl->copy_stream;
        if (known && pl->done_valid[slot]) {
            // the slot is free once the run two calls ago has finished; the previous run reads the other slot and
            // the partial rows behind both
            PS_CUDA_TRY(cudaStreamWaitEvent(cs, pl->ev_done[slot], 0));
        } else {
            // First use of this memory, slots that have moved, or another plan's work list in it: the upload is
            // ordered after everything already on the caller's stream (every earlier run that shares this workspace
            // is on that stream, or ordered before this call by the caller).
            PS_CUDA_TRY(cudaEventRecord(pl->ev_fence, s));
            PS_CUDA_TRY(cudaStreamWaitEvent(cs, pl->ev_fence, 0));
            if (!known) pl->done_valid[0] = pl->done_valid[1] = false;
        }
        PS_CUDA_TRY(cudaMemcpyAsync(ws, pl->pinned, pl->image_bytes, cudaMemcpyHostToDevice, cs));
        PS_CUDA_TRY(cudaEventRecord(pl->ev_copied[slot], cs));
        PS_CUDA_TRY(cudaStreamWaitEvent(s, pl->ev_copied[slot], 0));
        pl->copy_pending = true;
        pl->last_slot = slot;
    } else {
        PS_CUDA_TRY(cudaMemcpyAsync(ws, pl->pinned, pl->image_bytes, cudaMemcpyHostToDevice, s));
        PS_CUDA_TRY(cudaStreamSynchronize(s));  // no event to guard the staging image: finish the copy now
    }
    // the upload is in place (or queued): only now does the run count
    if (as_params) {
        if (pl->inline_runs == 0x1fffffffu) {  // tags begin again
            PS_CUDA_TRY(cudaMemsetAsync(own_hdr, 0, sizeof(WsHeader), s));
            pl->inline_runs = 0;
        }
        ++pl->inline_runs;
        pl->last_hdr = own_hdr;
        pl->last_tag = (int32_t)(pl->inline_runs << 2);
    } else {
        ++pl->run_no;
        pl->layout_moved = false;
        pl->last_ws = workspace_dev;
        pl->last_hdr = (WsHeader*)ws;
        pl->last_tag = 0;
        pl->done_valid[slot] = false;  // until this run's own completion event is recorded below
    }

    RunArgs a{};
    a.shape = pl->shape;
    a.pool = pool.base;
    a.num_pages = pool.num_pages;
    a.q = (const __nv_bfloat16*)q_dev;
    a.block_table = block_table_dev;
    a.max_pages = pl->max_pages;
    a.out = (__nv_bfloat16*)out_dev;
    a.lse = lse_out_dev;
    a.stream = s;
    a.num_sms = pl->num_sms;
    a.dec_sms = pl->dec_sms;
    a.pf_sms = pl->pf_sms;
    a.pairs = pl->pairs;
    a.dec_pages = pl->dec_pages;
    a.total_q = (int32_t)pl->info.total_q_tokens;
    a.n_req = pl->n;
    a.wait_limit_ns = pl->wait_limit_ns;
    a.early = !capturing;
    if (as_params) {
        a.inline_pieces = pl->pieces.data();
        a.inline_items = pl->prefill.empty() ? nullptr : pl->prefill.data();
        a.inline_starts = pl->prefill_cta_start.data();
    }
    a.tag = pl->last_tag;
    a.w.hdr = pl->last_hdr;
    a.w.pieces = (const DecodePiece*)(ws + pl->off_pieces);
    a.w.units = (const DecodeUnit*)(ws + pl->off_units);
    a.w.prefill = (const PrefillItem*)(ws + pl->off_prefill);
    a.w.merge = (const MergeEntry*)(ws + pl->off_merge);
    a.w.part_lse = (float*)(ws_base + pl->off_part_lse);
    a.w.part_o = (float*)(ws_base + pl->off_part_o);
    a.w.n_units = (int32_t)pl->units.size();
    a.w.n_cta_pieces = pl->cta_pieces ? (int32_t)pl->pieces.size() : 0;
    a.w.n_prefill = (int32_t)pl->prefill.size();
    a.w.n_merge = (int32_t)pl->merge.size();
    for (const MergeEntry& me : pl->merge) a.w.merge_segs = std::max(a.w.merge_segs, me.n_seg);
    a.w.n_dmerge = (int32_t)pl->dmerge.size();
    a.w.n_part_slots = pl->info.n_partial_slots;
    a.w.dmerge = (const DecodeMerge*)(ws + pl->off_dmerge);
    a.w.dmerge_cnt = (int32_t*)(ws + pl->off_dmerge_cnt);
    a.w.prefill_cta_start = (const int32_t*)(ws + pl->off_cta_start);
    a.w.n_prefill_ctas = pl->prefill_cta_start.empty() ? 0 : (int32_t)pl->prefill_cta_start.size() - 1;

    // events per recorded run: prefill begin/end, decode begin/end, merge begin/end
    const bool rec = !capturing && pl->timing && (size_t)(pl->timed_runs + 1) * 6 <= pl->tev.size();
    cudaEvent_t* ev = rec ? &pl->tev[(size_t)pl->timed_runs * 6] : nullptr;
    ps_status st = PS_OK;
    bool merged = false;  // the merge kernel has been launched already
    // dynamic item queue with more items than workers: the decode kernel's SMs help once it has ended
    const bool helpers = a.w.n_prefill_ctas == 0 && a.w.n_prefill > pl->pf_workers;
    if (pl->concurrent && !(rec && pl->side_stream) && (as_params || (!capturing && !helpers && !(pl->decode_last && a.w.n_merge > 0)))) {
        // Mixed batch: both kernels on the caller's stream, the prefill kernel launched as soon as the decode kernel has begun and
        // waiting for its end only at its own, and the merge kernel behind both.  (A second stream costs two events, which take
        // some 3 us each between kernels: tiny mixed batch 22.5 -> 16.8 us, with the list as parameters; 32 rows of 2048 tokens
        // beside a 512-token chunk 58.1 -> 57.2.)  On a second stream the merge kernel runs while the decode kernel still does: worth
        // more where that one ends last by 2.5 us and more (60 rows of 2500 tokens and 300 on 5000 114.2 / 107.7, 150 of 1500 and 300 on 5000
        // at 8 q / 2 kv heads 52.3 / 49.1, at head dimension 64 88.1 / 83.8; 58 batches 2 to 8 %), less where it does not (3 rows and 300 on
        // 5000 30.9 / 34.7, at head dimension 64 24.7 / 28.7; 200 batches up to 20 %).  Helpers have to start as soon as the decode kernel
        // ends, so batches with a queue keep the second stream.  So do runs that record events: one between the two launches would hold
        // the prefill kernel back until the decode kernel's end.
        RunArgs ad = a;
        ad.sm_pairs = pl->pf_workers < pl->pf_sms;
        if (rec) cudaEventRecord(ev[2], s);  // (without a second stream the kernels follow one another)
        st = launch_decode(ad);
        if (rec && st == PS_OK) cudaEventRecord(ev[3], s);
        if (rec && st == PS_OK) cudaEventRecord(ev[0], s);
        RunArgs ap = a;
        ap.beside = true;
        if (st == PS_OK) st = launch_prefill(ap);
        if (rec && st == PS_OK) cudaEventRecord(ev[1], s);
        if (st != PS_OK) return st;
    } else if (pl->concurrent && pl->side_stream) {
        // Mixed batch: the decode kernel runs on its share of the SMs on a second stream while the
        // prefill kernel runs on the rest.  Both need about 200 KB of shared memory per CTA, so each SM
        // holds one CTA of either kernel.
        cudaStream_t side = pl->side_stream;
        PS_CUDA_TRY(cudaEventRecord(pl->ev_fork, s));
        PS_CUDA_TRY(cudaStreamWaitEvent(side, pl->ev_fork, 0));
        // From here on the side stream belongs to this call (inside a capture: to the capture): whatever
        // fails below, it is joined back into the caller's stream before the call returns.
        if (rec) cudaEventRecord(ev[2], side);
        RunArgs ad = a;
        ad.sm_pairs = pl->pf_workers < pl->pf_sms;
        ad.stream = side;
        st = launch_decode(ad);
        if (rec && st == PS_OK) cudaEventRecord(ev[3], side);
        if (rec && st == PS_OK) cudaEventRecord(ev[0], s);
        if (st == PS_OK) st = launch_prefill(a);
        if (rec && st == PS_OK) cudaEventRecord(ev[1], s);
        if (st == PS_OK && !helpers) {
            // Only this launch writes prefill partials: combine them right behind it, on the SMs it leaves, while
            // the decode kernel is still streaming (decode rows are combined inside the decode kernel).
            // (not launched early: its CTAs, waiting beside the decode kernel's, slowed a batch of 48 decode rows and two chunks
            // at head dimension 64 from 70 to 81 us)
            RunArgs am = a;
            am.early = false;
            if (rec) cudaEventRecord(ev[4], s);
            st = launch_merge(am);
            if (rec) cudaEventRecord(ev[5], s);
            merged = true;
        }
        if (st == PS_OK && helpers) {
            // dynamic item queue: once the decode CTAs have left their SMs, as many more prefill CTAs
            // start there and help drain the same queue
            RunArgs ah = a;
            ah.stream = side;
            ah.pf_sms = a.dec_sms;
            ah.early = false;  // (waiting for the decode kernel it would hold SMs that the first launch needs)
            st = launch_prefill(ah);
        }
        const cudaError_t ej = cudaEventRecord(pl->ev_join, side);
        const cudaError_t ew = ej == cudaSuccess ? cudaStreamWaitEvent(s, pl->ev_join, 0) : ej;
        if (st != PS_OK) return st;
        PS_CUDA_TRY(ew);
    } else {
        if (rec) cudaEventRecord(ev[0], s);
        st = launch_prefill(a);
        if (st != PS_OK) return st;
        if (rec) cudaEventRecord(ev[1], s);
        if (rec) cudaEventRecord(ev[2], s);
        st = launch_decode(a);
        if (st != PS_OK) return st;
        if (rec) cudaEventRecord(ev[3], s);
    }
    if (!merged) {
        if (rec) cudaEventRecord(ev[4], s);
        st = launch_merge(a);
        if (rec) cudaEventRecord(ev[5], s);
    }
    if (rec) ++pl->timed_runs;
    if (pl->copy_stream && st == PS_OK && !capturing && !as_params) {
        PS_CUDA_TRY(cudaEventRecord(pl->ev_done[slot], s));
        pl->done_valid[slot] = true;
    }
    return st;
}

ps_status ps_plan_set_wait_limit(ps_plan* pl, int64_t limit_ns) {
    if (!pl) return fail(PS_ERR_INVALID, "null argument");
    if (limit_ns < 0 || limit_ns > kMaxWaitLimitNs)
        return fail(PS_ERR_INVALID, "limit_ns=%lld outside [0, %lld]", (long long)limit_ns, (long long)kMaxWaitLimitNs);
    pl->wait_limit_ns = limit_ns;
    return PS_OK;
}

ps_status ps_plan_set_timing(ps_plan* pl, int32_t max_runs) {
    if (!pl) return fail(PS_ERR_INVALID, "null argument");
    if (max_runs < 0 || max_runs > 4096) return fail(PS_ERR_INVALID, "max_runs=%d outside [0, 4096]", max_runs);
    pl->timed_runs = 0;
    pl->timing = max_runs > 0;
    while (pl->tev.size() < (size_t)max_runs * 6) {
        cudaEvent_t e;
        PS_CUDA_TRY(cudaEventCreate(&e));
        pl->tev.push_back(e);
    }
    return PS_OK;
}

ps_status ps_plan_get_timing(ps_plan* pl, void* stream, float* prefill_ms_out, float* decode_ms_out, float* merge_ms_out,
                             int32_t* n_runs_out) {
    if (!pl || !prefill_ms_out || !decode_ms_out || !merge_ms_out || !n_runs_out) return fail(PS_ERR_INVALID, "null argument");
    PS_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    double acc[3] = {0, 0, 0};
    for (int r = 0; r < pl->timed_runs; ++r)
        for (int k = 0; k < 3; ++k) {
            float ms = 0.f;
            PS_CUDA_TRY(cudaEventElapsedTime(&ms, pl->tev[(size_t)r * 6 + 2 * k], pl->tev[(size_t)r * 6 + 2 * k + 1]));
            acc[k] += ms;
        }
    const double n = pl->timed_runs > 0 ? pl->timed_runs : 1;
    *prefill_ms_out = (float)(acc[0] / n);
    *decode_ms_out = (float)(acc[1] / n);
    *merge_ms_out = (float)(acc[2] / n);
    *n_runs_out = pl->timed_runs;
    return PS_OK;
}

ps_status ps_plan_status(ps_plan* pl, void* stream) {
    if (!pl) return fail(PS_ERR_INVALID, "null argument");
    PS_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    if (!pl->last_hdr) return PS_OK;
    int32_t status = 0;
    PS_CUDA_TRY(cudaMemcpy(&status, &pl->last_hdr->status, sizeof status, cudaMemcpyDeviceToHost));
    status = (status & ~3) == pl->last_tag ? status & 3 : 0;  // (else an earlier run's)
    if (status & kStatusTimeout) return fail(PS_ERR_TIMEOUT, "a bounded device-side wait expired; output is invalid");
    if (status & kStatusBounds) return fail(PS_ERR_BOUNDS, "a block-table entry pointed outside the pool");
    return PS_OK;
}

}  // extern "C"

namespace ps {
size_t plan_workspace_bytes(const ps_plan* pl) { return pl ? pl->ws_bytes : 0; }
}  // namespace ps
