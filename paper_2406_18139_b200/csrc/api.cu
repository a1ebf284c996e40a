// Host side of the C ABI: argument checks, workspace carving, the request table, TMA tensor maps
// and the launch sequence.  Nothing here synchronises with the device or allocates device memory.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <initializer_list>
#include <functional>
#include <mutex>
#include <queue>
#include <vector>

#include <cudaTypedefs.h>

#include "internal.h"

namespace lookm {
namespace {

thread_local int g_launches = 0;
thread_local void* const* g_stage_events = nullptr;

// Records stage event i of the caller (if per-stage timing is on); errors are ignored on purpose:
// timing must never change the result of a call.
void mark_stage(int i, cudaStream_t st) {
    if (g_stage_events && g_stage_events[i]) cudaEventRecord(static_cast<cudaEvent_t>(g_stage_events[i]), st);
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct Plan {
    int n_req = 0, n_q_heads = 0, n_kv_heads = 0, group = 1;
    long long T = 0, sum_B = 0, sum_E = 0, sum_EB = 0;
    int max_L = 0, max_E = 0, max_B = 0;
    int n_none = 0;                         // requests with LOOKM_MERGE_NONE
    long long out_stride_head = 0;          // elements between heads of a single-prompt output
    int n_items[3] = {0, 0, 0};
    long long total_slots = 0;              // n_kv_heads * sum_B
    long long total_units = 0;              // merge work units
    std::vector<Req> reqs;                  // table order (longest first)
    std::vector<int> out_len;               // caller order
    // workspace offsets (bytes)
    int splits[2] = {1, 1};                 // ranges of a sweep 1 / sweep 2 item's streamed tiles
    int blocks = 1;                         // blocks per sweep item
    int tail_sets = 0, tail_begin = 0;      // several blocks per item: shortest sets that every request keeps
                                            // for the end, and the first item of these
    size_t n_arrived[2] = {0, 0};           // their arrival counters
    size_t clear_words = 64;                // status word and arrival counters
    size_t o_status, o_verdicts, o_reqs, o_lse, o_lse_split, o_scores, o_rank, o_rnorm_all, o_kept, o_evict, o_kept_keys,
        o_rnorm_kept, o_assign, o_sim, o_row_begin, o_entries, o_units, o_slot_cnt, o_parts, o_sort_a, o_sort_b,
        total;
};

struct DeviceInfo { int sms = 0; int cc_major = 0; bool ok = false; };
int device_info(DeviceInfo& out);

// Blocks per sweep item, from the scores of some 370 problems with one, two and four blocks per item (us).
// Several blocks pay where there are enough items and the items are full.
//   Two blocks, one prompt whose items stream 13 tiles on average, 16 with grouped heads: from 6.4 blocks per SM on (3200
// tokens x 32 heads, 5.4 per SM, 118 | 120, 2600 x 40, 5.7, 108 | 111, 3500 x 32, 6.1, 148 | 143, but a whole layer of it 221.8 | 223, at a
// higher clock, of 2800 x 40 189 | 196; 3800 x 32, 6.5, 165.8 | 162.2, 4096 x 32, 6.9, 189 | 184, 5000 x 32, 8.6, 290 |
// 278, 20000 x 8, 8.5, 991 | 952, 8192 x 32, 13.8, 714 | 672; grouped heads, layers: 6000 x 16 on 4, 5.1, 244 | 255, 4000 x 24
// on 6, 5.2, 180 | 183, 3300 x 40 on 10, 13.5 tiles, 7.0, 193 | 199, 3000 x 40 on 8, 12.5, 6.5, 183 | 172, 5000 x 24 on 6, 6.5,
// 255 | 251, 8000 x 16 on 4, 6.8, 388 | 372, 5000 x 32 on 8, 8.6, 324 | 314).  Calls in a row for some tenths of a second, which
// settle at the power limit: a few calls on a cool GPU are up to 4 % faster in single blocks from 6.4 to 8 per SM (layers, 12 ms | 500
// ms in a row, single - pairs: 17707 x 8, 7.5, 957 - 983 | 976 - 950, 4453 x 32 on 8, 7.6, 252 - 262 | 262 - 263).
// Shorter ones and two prompts: from nine (256 x 512, two tiles, 6.9, 36 | 42, 1000 x 128, five, 6.9, 67 | 70, 1200 x 96 on
// 48, six, 6.5, 71 | 78; layers of two of 2250 on average x 32, 7.6, 232 | 236).
//   More prompts, whose single blocks come out uneven from a fixed deal: from five (three of 900 x 32, 5.2, 66 |
// 58).  The items have to be three quarters full (93 of 128 tokens x 32: one block each, 111 | 135; 31 of 384: two
// items for three, 124 | 134).  Single blocks take the query heads of a group together in sweep 2, and the fixed
// deal evens out with many items, so grouped heads also need streamed tiles in an item: two on average below
// seven blocks per SM, two and a half below 24, else five (six of 400 x 32 on 8, three tiles, 5.2 per SM, 53 | 49, 40
// of them, 35 per SM, 219 | 246; 46 of 256, two tiles, 20 per SM, 100 | 114; 15 of 700, four tiles, 169 | 159).
//   Four blocks, one prompt: from four items per SM (9000 x 32, 3.9, 846 with two | 843, 8192 x 40, 4.3, 862 | 844,
// 16384 x 32, 6.9, 2662 | 2583).  More: from eight, with six streamed tiles each on average (five of 2000 x 32,
// 4.3 items, 257 | 276; 15 of 700, 6.5, 155 | 178; 32 of 33 to 2918 x 16, 11.4, 605 | 594).
int sweep_blocks(const Plan& pl, long long sms) {
    const auto shape = [&](int k, long long& sets, long long& streamed) {
        sets = streamed = 0;
        for (const Req& q : pl.reqs) {
            const long long n = (q.nblk + k - 1) / k;
            sets += n;
            streamed += n * q.nblk - k * n * (n - 1) / 2;            // a set streams the tiles from its first block on
        }
    };
    const bool one = pl.n_req == 1;
    long long blocks, sets, streamed;
    shape(1, blocks, streamed);
    shape(4, sets, streamed);
    if (sets * pl.n_q_heads >= (one ? 4 : 8) * sms && (one || streamed >= 6 * sets)) return 4;
    shape(2, sets, streamed);
    const long long all = blocks * pl.n_q_heads;
    const int half_tiles = pl.group == 1 ? 0 : all < 7 * sms ? 4 : all < 24 * sms ? 5 : 10;
    const bool many = 10 * all >= (one && streamed >= (pl.group == 1 ? 13 : 16) * sets ? 64 : pl.n_req <= 2 ? 90 : 50) * sms;
    return many && 100 * blocks >= 76 * 2 * sets && 2 * streamed >= half_tiles * sets ? 2 : 1;
}
// The kTailSets shortest items of all prompts come last: with each prompt's items in a row the last
// prompt's longest ones would end the sweep.  Scores of eight prompts of 4000 to 6000 tokens x 16 heads
// (8.6 items per SM), in rows | last: 1122 us | 1094, eight of 5000 x 16 1152 | 1051, four of 1000 to 12000 x 8
// 603 | 590, three of 2000 to 3000 x 32 291 | 285.  Neighbouring CTAs then share no tiles in L2, which costs more
// where there are many items: 16 prompts of 1000 to 3000 x 32 (14 per SM) 937 | 944, from 20 per SM no difference
// beyond the scatter.
constexpr int kTailSets = 6, kTailItemsPerSm = 12;
// Splits of the sweep items: as many as bring the longest item down to what an SM has on average, if it
// is more than one and a half times that and ten tiles longer.  Both sweeps together, us, whole | cut: 5000
// tokens with 2 heads 63.5 | 38, 12000 with 2 query on 1 KV head 188 | 110, 2048 with 32 on 8 78 | 63, 700
// with 32 on 8 35 | 25; ten tiles longer: 1300 x 1 23 | 18, 1300 x 4 23.7 | 22.3.  Nine: 1600 x 8 27 | 33, 2048 x 8 30 |
// 36, 2600 x 8 38 | 42: the partial results cost more than they save.
void plan_splits(Plan& pl) {
    DeviceInfo di;
    const long long sms = (device_info(di) == LOOKM_OK && di.sms > 0) ? di.sms : 148;
    long long tiles = 0, blocks = 0;
    for (const Req& q : pl.reqs) {
        tiles += (long long)q.nblk * (q.nblk + 1) / 2;
        blocks += (long long)q.nblk * pl.n_q_heads;
    }
    const long long mean = std::max<long long>(1, tiles * pl.n_q_heads / sms);
    pl.blocks = sweep_blocks(pl, sms);
    if (pl.blocks > 1) {
        if (blocks < kTailItemsPerSm * pl.blocks * sms)
            pl.tail_sets = std::min(kTailSets, (pl.reqs.back().nblk + pl.blocks - 1) / pl.blocks);
        return;
    }
    for (int s = 0; s < 2; ++s) {
        const long long longest = (long long)pl.reqs[0].nblk * (s ? pl.group : 1);
        if (2 * longest > 3 * mean && longest >= mean + 10)
            pl.splits[s] = (int)std::min<long long>(kMaxSplits, (longest + mean - 1) / mean);
    }
    // (sweep 1's partial results, 8 bytes per range, query head and token, have room where the kept keys go)
    pl.splits[0] = std::min(pl.splits[0], std::max(1, 2 * kHeadDim / (8 * pl.group)));
}

// Returns LOOKM_OK or the status describing the first bad argument.
int build_plan(Plan& pl, const lookm_layout* lay, int n_req, const int* cu_seqlens,
               const int* seq_lens, const int* budgets, const int* windows, const int* modes) {
    if (!lay || n_req <= 0 || (!cu_seqlens && !seq_lens)) return LOOKM_ERR_INVALID_ARG;
    if (lay->head_dim != kHeadDim) return LOOKM_ERR_UNSUPPORTED;
    if (lay->n_kv_heads <= 0 || lay->n_q_heads <= 0 || lay->n_q_heads % lay->n_kv_heads)
        return LOOKM_ERR_INVALID_ARG;
    if (lay->n_kv_heads > 65535 || n_req > 65535) return LOOKM_ERR_UNSUPPORTED;
    pl.n_req = n_req;
    pl.n_q_heads = lay->n_q_heads;
    pl.n_kv_heads = lay->n_kv_heads;
    pl.group = lay->n_q_heads / lay->n_kv_heads;
    pl.reqs.resize(n_req);
    pl.out_len.resize(n_req);
    long long tok = 0, out = 0, ev = 0, eb = 0;
    for (int r = 0; r < n_req; ++r) {
        const long long begin = cu_seqlens ? cu_seqlens[r] : tok;
        const long long L = cu_seqlens ? (long long)cu_seqlens[r + 1] - cu_seqlens[r] : seq_lens[r];
        if (begin != tok || L <= 0 || L > (1 << 30)) return LOOKM_ERR_INVALID_ARG;
        const int budget = budgets ? budgets[r] : (int)L;
        const int window = windows ? windows[r] : 0;
        const int mode = modes ? modes[r] : 0;
        if (budget <= 0 || window < 0 || mode < 0 || mode > LOOKM_MERGE_NONE) return LOOKM_ERR_INVALID_ARG;
        if (mode == LOOKM_MERGE_NONE) ++pl.n_none;
        Req& q = pl.reqs[r];
        q.tok_begin = (int)begin;
        q.L = (int)L;
        q.B = (int)std::min<long long>(budget, L);
        q.M = std::min(window, q.B);
        q.E = q.L - q.B;
        q.mode = mode;
        q.nblk = (q.L + kTile - 1) / kTile;
        q.out_begin = (int)out;
        q.kept_off = (long long)pl.n_kv_heads * out;
        q.ev_off = (long long)pl.n_kv_heads * ev;
        q.sim_off = (long long)pl.n_kv_heads * eb;
        q.rp_off = q.kept_off + (long long)pl.n_kv_heads * r;
        pl.out_len[r] = q.B;
        tok += L;
        out += q.B;
        ev += q.E;
        eb += (long long)q.E * q.B;
        pl.max_L = std::max(pl.max_L, q.L);
        pl.max_E = std::max(pl.max_E, q.E);
        pl.max_B = std::max(pl.max_B, q.B);
    }
    pl.T = tok;
    pl.sum_B = out;
    pl.sum_E = ev;
    pl.sum_EB = eb;
    pl.total_slots = (long long)pl.n_kv_heads * out;
    if (pl.T + kTile >= (1ll << 31) || pl.total_slots + kTile >= (1ll << 31) ||
        (long long)pl.n_q_heads * ((pl.T + kTile - 1) / kTile + n_req) >= (1ll << 31))
        return LOOKM_ERR_UNSUPPORTED;
    // table order: longest request first
    std::stable_sort(pl.reqs.begin(), pl.reqs.end(), [](const Req& a, const Req& b) { return a.L > b.L; });
    plan_splits(pl);
    long long it0 = 0, it1 = 0, it2 = 0, slots = 0, units = 0, tiles = 0;
    // Merge work units (the kernel reads n_kv_heads * T rows): every warp gets the same number of
    // units, one if that keeps a unit within kMaxUnitEntries rows.  The units of a request are laid
    // out heads fastest, so a wave of warps reads one token window of all heads; with very long
    // units (a batch of many prompts) every warp would stream a far-away window of its own, and a
    // unit count just above the warp count would leave a second, nearly empty wave.
    int unit_entries = kMinUnitEntries;
    {
        DeviceInfo di;
        const int sms = (device_info(di) == LOOKM_OK && di.sms > 0) ? di.sms : 148;
        const long long per_warp = ((long long)pl.n_kv_heads * pl.T) / ((long long)sms * merge_warps_per_sm());
        if (per_warp > unit_entries) {
            const long long per_warp_units = (per_warp + kMaxUnitEntries - 1) / kMaxUnitEntries;
            const long long rows = (per_warp + per_warp_units - 1) / per_warp_units;
            unit_entries = (int)std::max<long long>(kMinUnitEntries, (rows + 7) / 8 * 8);
        }
    }
    for (Req& q : pl.reqs) {
        q.item_begin[kSweep1] = (int)it0;
        q.item_begin[kSweep2] = (int)it1;
        q.item_begin[kMatch] = (int)it2;
        q.slot_begin = (int)slots;
        q.unit_begin = (int)units;
        q.unit_entries = unit_entries;
        q.tile_begin = (int)tiles;
        tiles += q.nblk;
        const bool merges = q.mode != LOOKM_MERGE_NONE;
        const long long n_units = merges ? (q.L + unit_entries - 1) / unit_entries : 0;
        units += (long long)pl.n_kv_heads * n_units;
        const long long sets = (q.nblk + pl.blocks - 1) / pl.blocks - pl.tail_sets;
        it0 += sets * pl.n_q_heads * pl.splits[0];
        // (several blocks per item: the query heads of a group are items of their own in sweep 2 too)
        it1 += sets * (pl.blocks > 1 ? pl.n_q_heads : pl.n_kv_heads) * pl.splits[1];
        // match items: blocks of 128 entries of every head's evicted list
        it2 += (q.E > 0 && merges) ? (long long)((q.E + kTile - 1) / kTile) * pl.n_kv_heads : 0;
        slots += (long long)q.B * pl.n_kv_heads;
    }
    pl.total_units = units;
    pl.tail_begin = (int)it0;                       // (the same in both sweeps: see above)
    pl.n_items[kSweep1] = (int)(it0 + (long long)pl.tail_sets * n_req * pl.n_q_heads);
    pl.n_items[kSweep2] = (int)(it1 + (long long)pl.tail_sets * n_req * pl.n_q_heads);
    pl.n_items[kMatch] = (int)it2;

    size_t o = 0;
    auto carve = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    const size_t Hq = pl.n_q_heads, Hkv = pl.n_kv_heads, T = (size_t)pl.T;
    // Every list is sized for the worst case over budgets (at most T kept and T evicted rows per
    // head) and over how the sweeps are cut, so the carving depends only on the prompt lengths and head
    // counts and never shrinks with more query heads: a size computed for a layout also serves the entry
    // points that know its KV heads alone.
    const size_t score_parts = pl.blocks > 1 ? pl.group : pl.splits[1];       // partial column sums of sweep 2
    for (int s = 0; s < 2; ++s)
        if (pl.splits[s] > 1 || (s && score_parts > 1)) pl.n_arrived[s] = 4 * (size_t)tiles * (s ? Hkv : Hq);
    pl.clear_words += pl.n_arrived[0] + pl.n_arrived[1];
    pl.o_status = carve(4 * (64 + 4 * (size_t)tiles * (Hq + Hkv)));
    // (where sweep 1 leaves verdicts, one per CTA and so at most tiles * Hq, its items are whole and need no counters)
    pl.o_verdicts = pl.o_status + 4 * (64 + 4 * (size_t)tiles * Hkv);
    pl.o_reqs = carve(sizeof(Req) * n_req);
    pl.o_lse = carve(4 * Hq * T);
    pl.o_lse_split = carve(32 * Hq * T);
    pl.o_scores = carve(4 * Hkv * T);
    pl.o_rank = carve(4 * Hkv * T);
    pl.o_rnorm_all = carve(4 * Hkv * T);
    pl.o_kept = carve(4 * Hkv * T);
    pl.o_evict = carve(4 * Hkv * T);
    // The kept keys are gathered after both sweeps are done; until then their place holds the sweeps'
    // partial results: sweep 1's ranges (see plan_splits), sweep 2's ranges or query heads of a group.
    pl.o_kept_keys = carve(std::max(2 * (size_t)kHeadDim * Hkv * T, 4 * Hq * T));
    pl.o_rnorm_kept = carve(4 * Hkv * T);
    pl.o_assign = carve(4 * Hkv * T);
    pl.o_sim = carve(4 * Hkv * T);
    pl.o_row_begin = carve(4 * (Hkv * T + Hkv * (size_t)n_req));
    pl.o_entries = carve(8 * Hkv * T);
    pl.o_units = carve(16 * (size_t)pl.total_units);
    pl.o_slot_cnt = carve(4 * Hkv * T);
    pl.o_parts = carve((size_t)kMergePartBytes * (size_t)pl.total_units);
    pl.o_sort_a = carve(8 * Hkv * T);
    pl.o_sort_b = carve(8 * Hkv * T);
    pl.total = o;
    return LOOKM_OK;
}

int check_layout_ptrs(const lookm_layout* lay, const void* q, const void* k, const void* v) {
    auto bad_ptr = [](const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 15u); };
    if (bad_ptr(q) || bad_ptr(k) || bad_ptr(v)) return LOOKM_ERR_INVALID_ARG;
    if (lay->q_stride_tok % 8 || lay->q_stride_head % 8 || lay->kv_stride_tok % 8 ||
        lay->kv_stride_head % 8)
        return LOOKM_ERR_INVALID_ARG;
    if (lay->q_stride_tok <= 0 || lay->q_stride_head <= 0 || lay->kv_stride_tok <= 0 ||
        lay->kv_stride_head <= 0)
        return LOOKM_ERR_INVALID_ARG;
    // the merge kernel keeps the byte stride between tokens in 32 bits
    if (lay->kv_stride_tok >= (1ll << 31)) return LOOKM_ERR_UNSUPPORTED;
    if (!(lay->softmax_scale >= 0.f) || !std::isfinite(lay->softmax_scale)) return LOOKM_ERR_INVALID_ARG;
    return LOOKM_OK;
}

int check_workspace(const Plan& pl, void* ws, size_t bytes) {
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return LOOKM_ERR_INVALID_ARG;
    if (bytes < pl.total) return LOOKM_ERR_WORKSPACE_TOO_SMALL;
    return LOOKM_OK;
}

// ---- device facts and the tensor-map encoder ---------------------------------------------------
int device_info(DeviceInfo& out) {
    static std::mutex mu;
    static DeviceInfo cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LOOKM_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!cache[dev].ok) {
        if (cudaDeviceGetAttribute(&cache[dev].sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&cache[dev].cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
            return LOOKM_ERR_CUDA;
        cache[dev].ok = true;
    }
    out = cache[dev];
    return out.cc_major == 10 ? LOOKM_OK : LOOKM_ERR_UNSUPPORTED;
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// bf16 tensor [tokens, heads, 128] with element strides; box = 128 tokens x 1 head x 64 features
// (128 bytes) with the 128-byte swizzle; out-of-range rows read as zero.
int make_map_3d(CUtensorMap* map, const void* base, long long tokens, int heads,
                long long stride_tok, long long stride_head) {
    auto enc = tensor_map_encoder();
    if (!enc) return LOOKM_ERR_CUDA;
    cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)heads, (cuuint64_t)tokens};
    cuuint64_t strides[2] = {(cuuint64_t)stride_head * 2, (cuuint64_t)stride_tok * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)kTile};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LOOKM_OK : LOOKM_ERR_CUDA;
}

// The 16-column companion of the query tensor ([tokens, heads, 16] bf16, 32-byte rows): boxes of
// 128 tokens of one head with the 32-byte swizzle.
int make_map_split(CUtensorMap* map, const void* base, long long tokens, int heads) {
    auto enc = tensor_map_encoder();
    if (!enc) return LOOKM_ERR_CUDA;
    cuuint64_t dims[3] = {16, (cuuint64_t)heads, (cuuint64_t)tokens};
    cuuint64_t strides[2] = {32, (cuuint64_t)heads * 32};
    cuuint32_t box[3] = {16, 1, (cuuint32_t)kTile};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LOOKM_OK : LOOKM_ERR_CUDA;
}

int make_map_2d(CUtensorMap* map, const void* base, long long rows) {
    auto enc = tensor_map_encoder();
    if (!enc) return LOOKM_ERR_CUDA;
    cuuint64_t dims[2] = {(cuuint64_t)kHeadDim, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kHeadDim * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                     box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? LOOKM_OK : LOOKM_ERR_CUDA;
}

#define LOOKM_CUDA(expr)                                  \
    do {                                                  \
        if ((expr) != cudaSuccess) return LOOKM_ERR_CUDA; \
    } while (0)
#define LOOKM_TRY(expr)                   \
    do {                                  \
        int st_ = (expr);                 \
        if (st_ != LOOKM_OK) return st_;  \
    } while (0)

// A whole-path call of one prompt in single blocks needs no table writer: its launches carry the request, and the
// first of them (sweep 1, or the one that takes its place) clears the words that later ones count in and writes the
// request to its row, for the launch that reads it there.
// (Eviction alone, and scores from a given log-sum-exp by themselves, keep it: their callers count five and three launches.)
bool first_launch_clears(const Plan& pl) { return pl.n_req == 1 && pl.blocks == 1 && pl.splits[0] == 1 && pl.n_none == 0; }

template <class T>
T* at(void* ws, size_t off) { return reinterpret_cast<T*>(static_cast<char*>(ws) + off); }

// Clears the status word and the arrival counters and writes the request table into the workspace (unless the
// call's first launch does what is needed of that).
int begin_call(const Plan& pl, void* ws, cudaStream_t st, bool first_clears = false) {
    g_launches = 0;
    if (first_clears) return LOOKM_OK;
    for (int base = 0; base < pl.n_req; base += kReqChunk) {
        ReqChunk chunk;
        const int cnt = std::min(kReqChunk, pl.n_req - base);
        std::memset(&chunk, 0, sizeof(chunk));
        std::memcpy(chunk.r, pl.reqs.data() + base, sizeof(Req) * cnt);
        LOOKM_CUDA(launch_write_table(chunk, cnt, at<Req>(ws, pl.o_reqs) + base, at<int>(ws, pl.o_status),
                                      base == 0 ? pl.clear_words : 0, st));
        ++g_launches;
    }
    return LOOKM_OK;
}

float scale_log2(const lookm_layout* lay) {
    const float s = lay->softmax_scale > 0.f ? lay->softmax_scale : 1.0f / std::sqrt((float)lay->head_dim);
    return s * 1.4426950408889634f;
}

ReqTable req_table(const Plan& pl, void* ws) {
    ReqTable t;
    t.rows = at<Req>(ws, pl.o_reqs);
    t.n = pl.n_req;
    t.only = pl.reqs[0];
    return t;
}

TileParams tile_params(const Plan& pl, void* ws, const lookm_layout* lay) {
    TileParams p;
    std::memset(&p, 0, sizeof(p));
    p.reqs = req_table(pl, ws);
    p.n_q_heads = pl.n_q_heads;
    p.n_kv_heads = pl.n_kv_heads;
    p.group = pl.group;
    p.T = pl.T;
    p.scale_log2 = scale_log2(lay);
    p.status = at<int>(ws, pl.o_status);
    p.blocks = pl.blocks;
    p.tail_begin = pl.tail_begin;
    p.tail_sets = pl.tail_sets;
    return p;
}

int run_score(const Plan& pl, const DeviceInfo& di, const lookm_layout* lay, const void* q,
              const void* k, float* scores, float* lse, bool lse_is_input, bool clears, void* ws, cudaStream_t st) {
    CUtensorMap map_q, map_k;
    LOOKM_TRY(make_map_3d(&map_q, q, pl.T, pl.n_q_heads, lay->q_stride_tok, lay->q_stride_head));
    LOOKM_TRY(make_map_3d(&map_k, k, pl.T, pl.n_kv_heads, lay->kv_stride_tok, lay->kv_stride_head));
    CUtensorMap map_x;
    unsigned short* split = at<unsigned short>(ws, pl.o_lse_split);
    LOOKM_TRY(make_map_split(&map_x, split, pl.T, pl.n_q_heads));
    TileParams p = tile_params(pl, ws, lay);
    p.lse = lse;
    p.lse_split = split;
    p.scores = scores;
    if (!lse_is_input) {
        p.n_items = pl.n_items[kSweep1];
        p.n_clear = clears ? (int)pl.clear_words : 0;
        p.verdicts = at<int>(ws, pl.o_verdicts);
        p.next_item = p.status + 16 + kSweep1;
        p.splits = pl.splits[0];
        p.parts1 = at<float2>(ws, pl.o_kept_keys);
        p.arrived = p.status + 64;
        LOOKM_CUDA(launch_tile_kernel(kSweep1, map_q, map_k, nullptr, p, di.sms, st));
        ++g_launches;
    } else {
        LOOKM_CUDA(launch_lse_split(lse, pl.n_q_heads, pl.T, p.scale_log2, split, p.reqs, p.status, clears ? (int)pl.clear_words : 0, st));
        ++g_launches;
    }
    mark_stage(1, st);
    p.n_verdicts = !lse_is_input && clears ? tile_grid(pl.n_items[kSweep1], di.sms) : 0;
    p.n_items = pl.n_items[kSweep2];
    p.next_item = p.status + 16 + kSweep2;
    p.splits = pl.splits[1];
    p.parts2 = at<float>(ws, pl.o_kept_keys);
    p.arrived = p.status + 64 + pl.n_arrived[0];
    LOOKM_CUDA(launch_tile_kernel(kSweep2, map_k, map_q, &map_x, p, di.sms, st));
    ++g_launches;
    mark_stage(2, st);
    return LOOKM_OK;
}

// norms_done: 1 / |k| of every key row is already in the workspace (written by the selection launch)
int run_match(const Plan& pl, const DeviceInfo& di, const lookm_layout* lay, const void* k,
              const int* kept_idx, const int* evict_idx, int* assign, float* sim, void* ws,
              bool norms_done, cudaStream_t st) {
    if (pl.n_items[kMatch] == 0) { mark_stage(4, st); mark_stage(5, st); return LOOKM_OK; }
    float* rnorm_all = at<float>(ws, pl.o_rnorm_all);
    float* rnorm_kept = at<float>(ws, pl.o_rnorm_kept);
    void* kept_keys = at<void>(ws, pl.o_kept_keys);
    const ReqTable reqs = req_table(pl, ws);
    if (!norms_done) {
        LOOKM_CUDA(launch_key_norms(k, lay->kv_stride_tok, lay->kv_stride_head, pl.n_kv_heads, pl.T,
                                    rnorm_all, st));
        ++g_launches;
    }
    LOOKM_CUDA(launch_gather_kept(k, lay->kv_stride_tok, lay->kv_stride_head, reqs,
                                  pl.n_kv_heads, pl.T, pl.total_slots, kept_idx, rnorm_all,
                                  kept_keys, rnorm_kept, at<int>(ws, pl.o_status), st));
    ++g_launches;
    mark_stage(4, st);
    CUtensorMap map_c;                           // the evicted rows are gathered, not tiled
    LOOKM_TRY(make_map_2d(&map_c, kept_keys, pl.total_slots));
    TileParams p = tile_params(pl, ws, lay);
    p.n_items = pl.n_items[kMatch];
    p.evict_idx = evict_idx;
    p.k_rows = k;
    p.k_stride_tok = lay->kv_stride_tok;
    p.k_stride_head = lay->kv_stride_head;
    p.rnorm_all = rnorm_all;
    p.rnorm_kept = rnorm_kept;
    p.assign = assign;
    p.sim = sim;
    LOOKM_CUDA(launch_match(map_c, p, di.sms, st));
    ++g_launches;
    mark_stage(5, st);
    return LOOKM_OK;
}

// The inversion's CTAs (kInvMaxCluster at most per request and head) run all at once, two per SM if their
// shared memory allows, and each gets kInvMinShare evicted tokens at least.
constexpr long long kInvCtasPerSm = 2, kInvSmemPerSm = 220 << 10;
constexpr int kInvMinShare = 512;
cudaError_t run_inversion(const Plan& pl, const DeviceInfo& di, const int* kept_idx, const int* evict_idx, const int* assign,
                          const float* sim, void* ws, cudaStream_t st) {
    const ReqTable reqs = req_table(pl, ws);
    int *status = at<int>(ws, pl.o_status), *row_begin = at<int>(ws, pl.o_row_begin);
    int2* entries = at<int2>(ws, pl.o_entries);
    int4* units = at<int4>(ws, pl.o_units);
    int* slot_cnt = at<int>(ws, pl.o_slot_cnt);
    const auto ctas_per_head = [&](long long per_sm) {
        int ctas = 1;
        while (ctas < kInvMaxCluster && 2ll * ctas * pl.n_kv_heads * pl.n_req <= per_sm * di.sms &&
               pl.max_E >= 2 * ctas * kInvMinShare)
            ctas *= 2;
        return ctas;
    };
    // counting, where it fits: a count per slot and warp in shared memory, a warp's rows in registers and
    // their counts in bytes (42 us sorted, 25 counted for 26214 evicted rows x 8 heads and 6554 slots)
    const long long slot_bytes = (long long)(pl.max_B + 4 * kInvMaxCluster) * kCountSlotBytes;
    int ctas = ctas_per_head(std::min(kInvCtasPerSm, std::max(1ll, kInvSmemPerSm / slot_bytes)));
    if (pl.max_B <= kCountMaxSlots && pl.max_E <= ctas * kCountWarps * kCountSeg) {
        const int max_slots = ctas * (((pl.max_B + ctas - 1) / ctas + 3) / 4 * 4);
        return launch_invert_counting(assign, kept_idx, evict_idx, sim, reqs, pl.n_kv_heads, ctas, max_slots, pl.T,
                                      entries, units, slot_cnt, status, st);
    }
    // counter width and widest digit over the requests of the call
    ctas = ctas_per_head(kInvCtasPerSm);
    const bool wide = pl.max_E > kInvWideCountsAbove;
    int digit_bits = 1;
    for (const Req& r : pl.reqs) {
        int n_pass, dbits;
        invert_digits(r.B, wide ? kInvDigitBits32 : kInvDigitBits16, n_pass, dbits);
        digit_bits = std::max(digit_bits, dbits);
    }
    return launch_invert_assignment(assign, kept_idx, evict_idx, sim, reqs, pl.n_kv_heads, ctas, pl.T, wide, digit_bits, row_begin,
                                    entries, units, slot_cnt, at<unsigned>(ws, pl.o_sort_a), at<unsigned>(ws, pl.o_sort_b),
                                    status, st);
}

int run_merge(const Plan& pl, const lookm_layout* lay, const void* k, const void* v,
              const int* kept_idx, const int* evict_idx, const int* assign, const float* sim,
              int varlen_output, void* out_k, void* out_v, void* ws, cudaStream_t st) {
    const ReqTable reqs = req_table(pl, ws);
    int* status = at<int>(ws, pl.o_status);
    const bool short_merge = pl.max_L <= kMergeShortMax;
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    if (pl.n_none < pl.n_req && !short_merge) {
        LOOKM_CUDA(run_inversion(pl, di, kept_idx, evict_idx, assign, sim, ws, st));
        ++g_launches;
    }
    mark_stage(6, st);
    if (pl.n_none < pl.n_req) {
        if (short_merge)
            LOOKM_CUDA(launch_merge_short(k, v, lay->kv_stride_tok, lay->kv_stride_head, assign, kept_idx, evict_idx, sim,
                                          reqs, pl.n_kv_heads, pl.max_L, pl.max_E, pl.max_B, varlen_output,
                                          pl.out_stride_head, out_k, out_v, status, di.sms, st));
        else
            LOOKM_CUDA(launch_merge(k, v, lay->kv_stride_tok, lay->kv_stride_head, reqs,
                                    pl.n_kv_heads, pl.T, pl.total_units, at<int2>(ws, pl.o_entries),
                                    at<int4>(ws, pl.o_units), at<int>(ws, pl.o_slot_cnt),
                                    at<float>(ws, pl.o_parts), varlen_output, pl.out_stride_head, out_k,
                                    out_v, di.sms, st));
        ++g_launches;
    }
    if (pl.n_none > 0) {
        // eviction alone: the kept rows of those requests go straight to the output
        LOOKM_CUDA(launch_compact_kept(k, v, lay->kv_stride_tok, lay->kv_stride_head, reqs,
                                       pl.n_kv_heads, pl.total_slots, kept_idx, varlen_output,
                                       pl.out_stride_head, out_k, out_v, status, st));
        ++g_launches;
    }
    mark_stage(7, st);
    return LOOKM_OK;
}

// Output pointers are written with 16-byte stores, index and weight lists read as 32-bit words.
int check_out_ptrs(const void* out_k, const void* out_v) {
    if ((reinterpret_cast<uintptr_t>(out_k) & 15u) || (reinterpret_cast<uintptr_t>(out_v) & 15u))
        return LOOKM_ERR_INVALID_ARG;
    return LOOKM_OK;
}
int check_word_ptrs(std::initializer_list<const void*> ptrs) {
    for (const void* p : ptrs)
        if (reinterpret_cast<uintptr_t>(p) & 3u) return LOOKM_ERR_INVALID_ARG;
    return LOOKM_OK;
}

// Stride between the heads of a single-prompt output (0 = dense).
int set_out_stride(Plan& pl, int varlen_output, long long out_stride_head) {
    pl.out_stride_head = 0;
    if (varlen_output) return out_stride_head ? LOOKM_ERR_INVALID_ARG : LOOKM_OK;
    const long long dense = (long long)pl.out_len[0] * kHeadDim;
    if (out_stride_head == 0) { pl.out_stride_head = dense; return LOOKM_OK; }
    if (out_stride_head % 8 || out_stride_head < dense) return LOOKM_ERR_INVALID_ARG;
    pl.out_stride_head = out_stride_head;
    return LOOKM_OK;
}

int compress_common(const void* q, const void* k, const void* v, const uint8_t* mask,
                    const int* cu_seqlens, int n_req, const int* budgets, const int* windows,
                    const int* modes, const lookm_layout* lay, const lookm_options* opt,
                    int varlen_output, void* out_k, void* out_v, int* out_cu, void* ws,
                    size_t ws_bytes, void* stream) {
    const unsigned flags = opt ? opt->flags : 0u;
    const float* lse_in = opt ? opt->lse : nullptr;
    if (flags & ~LOOKM_OPT_NO_TEXT_PRIOR) return LOOKM_ERR_INVALID_ARG;
    const bool text_prior = !(flags & LOOKM_OPT_NO_TEXT_PRIOR);
    if (!q || !k || !v || (!mask && text_prior) || !out_k || !out_v || !budgets || !windows || !modes)
        return LOOKM_ERR_INVALID_ARG;
    Plan pl;
    LOOKM_TRY(build_plan(pl, lay, n_req, cu_seqlens, nullptr, budgets, windows, modes));
    LOOKM_TRY(check_layout_ptrs(lay, q, k, v));
    LOOKM_TRY(check_out_ptrs(out_k, out_v));
    LOOKM_TRY(check_word_ptrs({lse_in}));
    LOOKM_TRY(set_out_stride(pl, varlen_output, opt ? opt->out_stride_head : 0));
    LOOKM_TRY(check_workspace(pl, ws, ws_bytes));
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (out_cu) {
        out_cu[0] = 0;
        for (int r = 0; r < n_req; ++r) out_cu[r + 1] = out_cu[r] + pl.out_len[r];
    }
    const bool clears = first_launch_clears(pl);
    LOOKM_TRY(begin_call(pl, ws, st, clears));
    mark_stage(0, st);
    float* scores = at<float>(ws, pl.o_scores);
    int* kept = at<int>(ws, pl.o_kept);
    int* evict = at<int>(ws, pl.o_evict);
    int* rank = at<int>(ws, pl.o_rank);
    int* assign = at<int>(ws, pl.o_assign);
    float* sim = at<float>(ws, pl.o_sim);
    // a caller's log-sum-exp (read only) replaces the first sweep
    float* lse = lse_in ? const_cast<float*>(lse_in) : at<float>(ws, pl.o_lse);
    LOOKM_TRY(run_score(pl, di, lay, q, k, scores, lse, lse_in != nullptr, clears, ws, st));
    // the selection launch also computes the key norms that the matching needs
    const bool need_match = pl.n_items[kMatch] > 0;
    LOOKM_CUDA(launch_select(scores, text_prior ? mask : nullptr, req_table(pl, ws),
                             pl.n_kv_heads, pl.T, pl.max_L, kept, evict, rank, need_match ? k : nullptr,
                             lay->kv_stride_tok, lay->kv_stride_head, at<float>(ws, pl.o_rnorm_all),
                             di.sms, st));
    ++g_launches;
    mark_stage(3, st);
    LOOKM_TRY(run_match(pl, di, lay, k, kept, evict, assign, sim, ws, true, st));
    LOOKM_TRY(run_merge(pl, lay, k, v, kept, evict, assign, sim, varlen_output, out_k, out_v, ws, st));
    return LOOKM_OK;
}

}  // namespace
}  // namespace lookm

using namespace lookm;

extern "C" {

size_t lookm_workspace_size(const lookm_layout* layout, int n_requests, const int* seq_lens_host,
                            const int* budgets_host) {
    Plan pl;
    if (!seq_lens_host) return 0;
    if (build_plan(pl, layout, n_requests, nullptr, seq_lens_host, budgets_host, nullptr, nullptr) != LOOKM_OK)
        return 0;
    return pl.total;
}

int lookm_workspace_layout(const lookm_layout* layout, int n_requests, const int* seq_lens_host,
                           lookm_workspace_offsets* offsets_host) {
    Plan pl;
    if (!seq_lens_host || !offsets_host) return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(build_plan(pl, layout, n_requests, nullptr, seq_lens_host, nullptr, nullptr, nullptr));
    offsets_host->status = pl.o_status;
    offsets_host->lse = pl.o_lse;
    offsets_host->scores = pl.o_scores;
    offsets_host->rank = pl.o_rank;
    offsets_host->kept_idx = pl.o_kept;
    offsets_host->evict_idx = pl.o_evict;
    offsets_host->assign = pl.o_assign;
    offsets_host->sim = pl.o_sim;
    return LOOKM_OK;
}

int lookm_compress_layer_opt(const void* q, const void* k, const void* v, const uint8_t* modality_mask,
                             int seq_len, int budget, int recent_window, int merge_mode,
                             const lookm_layout* layout, const lookm_options* options, void* out_k,
                             void* out_v, int* out_len_host, void* workspace, size_t workspace_bytes,
                             void* cuda_stream) {
    if (seq_len <= 0) return LOOKM_ERR_INVALID_ARG;
    const int cu[2] = {0, seq_len};
    int out_cu[2] = {0, 0};
    const int st = compress_common(q, k, v, modality_mask, cu, 1, &budget, &recent_window, &merge_mode,
                                   layout, options, 0, out_k, out_v, out_cu, workspace, workspace_bytes,
                                   cuda_stream);
    if (st == LOOKM_OK && out_len_host) *out_len_host = out_cu[1];
    return st;
}

int lookm_compress_layer(const void* q, const void* k, const void* v, const uint8_t* modality_mask,
                         int seq_len, int budget, int recent_window, int merge_mode,
                         const lookm_layout* layout, void* out_k, void* out_v, int* out_len_host,
                         void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return lookm_compress_layer_opt(q, k, v, modality_mask, seq_len, budget, recent_window, merge_mode,
                                    layout, nullptr, out_k, out_v, out_len_host, workspace,
                                    workspace_bytes, cuda_stream);
}

int lookm_compress_varlen_opt(const void* q, const void* k, const void* v, const uint8_t* modality_mask,
                              const int* cu_seqlens_host, int n_requests, const int* budgets_host,
                              const int* windows_host, const int* merge_modes_host,
                              const lookm_layout* layout, const lookm_options* options, void* out_k,
                              void* out_v, int* out_cu_seqlens_host, void* workspace,
                              size_t workspace_bytes, void* cuda_stream) {
    if (!cu_seqlens_host) return LOOKM_ERR_INVALID_ARG;
    return compress_common(q, k, v, modality_mask, cu_seqlens_host, n_requests, budgets_host,
                           windows_host, merge_modes_host, layout, options, 1, out_k, out_v,
                           out_cu_seqlens_host, workspace, workspace_bytes, cuda_stream);
}

int lookm_compress_varlen(const void* q, const void* k, const void* v, const uint8_t* modality_mask,
                          const int* cu_seqlens_host, int n_requests, const int* budgets_host,
                          const int* windows_host, const int* merge_modes_host,
                          const lookm_layout* layout, void* out_k, void* out_v,
                          int* out_cu_seqlens_host, void* workspace, size_t workspace_bytes,
                          void* cuda_stream) {
    return lookm_compress_varlen_opt(q, k, v, modality_mask, cu_seqlens_host, n_requests, budgets_host,
                                     windows_host, merge_modes_host, layout, nullptr, out_k, out_v,
                                     out_cu_seqlens_host, workspace, workspace_bytes, cuda_stream);
}

int lookm_score(const void* q, const void* k, const int* cu_seqlens_host, int n_requests,
                const lookm_layout* layout, float* scores, float* lse, int lse_is_input,
                void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!q || !k || !cu_seqlens_host || !scores || (lse_is_input && !lse)) return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_word_ptrs({scores, lse}));
    Plan pl;
    LOOKM_TRY(build_plan(pl, layout, n_requests, cu_seqlens_host, nullptr, nullptr, nullptr, nullptr));
    LOOKM_TRY(check_layout_ptrs(layout, q, k, nullptr));
    LOOKM_TRY(check_workspace(pl, workspace, workspace_bytes));
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const bool clears = !lse_is_input && first_launch_clears(pl);
    LOOKM_TRY(begin_call(pl, workspace, st, clears));
    float* lse_buf = lse ? lse : at<float>(workspace, pl.o_lse);
    return run_score(pl, di, layout, q, k, scores, lse_buf, lse_is_input != 0, clears, workspace, st);
}

int lookm_select(const float* scores, const uint8_t* modality_mask, const int* cu_seqlens_host,
                 int n_requests, const int* budgets_host, const int* windows_host, int n_kv_heads,
                 int* kept_idx, int* evict_idx, int* rank, void* workspace, size_t workspace_bytes,
                 void* cuda_stream) {
    if (!scores || !cu_seqlens_host || !budgets_host || !windows_host || !kept_idx || !evict_idx)
        return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_word_ptrs({scores, kept_idx, evict_idx, rank}));
    lookm_layout lay;
    std::memset(&lay, 0, sizeof(lay));
    lay.n_q_heads = lay.n_kv_heads = n_kv_heads;
    lay.head_dim = kHeadDim;
    Plan pl;
    LOOKM_TRY(build_plan(pl, &lay, n_requests, cu_seqlens_host, nullptr, budgets_host, windows_host, nullptr));
    LOOKM_TRY(check_workspace(pl, workspace, workspace_bytes));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    LOOKM_TRY(begin_call(pl, workspace, st));
    LOOKM_CUDA(launch_select(scores, modality_mask, req_table(pl, workspace),
                             pl.n_kv_heads, pl.T, pl.max_L, kept_idx, evict_idx, rank, nullptr, 0, 0, nullptr, 0, st));
    ++g_launches;
    return LOOKM_OK;
}

int lookm_match(const void* k, const int* kept_idx, const int* evict_idx, const int* cu_seqlens_host,
                int n_requests, const int* budgets_host, const lookm_layout* layout, int* assign,
                float* sim, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!k || !kept_idx || !evict_idx || !cu_seqlens_host || !budgets_host || !assign || !sim)
        return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_word_ptrs({kept_idx, evict_idx, assign, sim}));
    Plan pl;
    LOOKM_TRY(build_plan(pl, layout, n_requests, cu_seqlens_host, nullptr, budgets_host, nullptr, nullptr));
    LOOKM_TRY(check_layout_ptrs(layout, nullptr, k, nullptr));
    LOOKM_TRY(check_workspace(pl, workspace, workspace_bytes));
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    LOOKM_TRY(begin_call(pl, workspace, st));
    return run_match(pl, di, layout, k, kept_idx, evict_idx, assign, sim, workspace, false, st);
}

int lookm_match_from_sim(const float* sim_matrix, const int* cu_seqlens_host, int n_requests,
                         const int* budgets_host, int n_kv_heads, int* assign, float* sim,
                         void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!sim_matrix || !cu_seqlens_host || !budgets_host || !assign || !sim) return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_word_ptrs({sim_matrix, assign, sim}));
    lookm_layout lay;
    std::memset(&lay, 0, sizeof(lay));
    lay.n_q_heads = lay.n_kv_heads = n_kv_heads;
    lay.head_dim = kHeadDim;
    Plan pl;
    LOOKM_TRY(build_plan(pl, &lay, n_requests, cu_seqlens_host, nullptr, budgets_host, nullptr, nullptr));
    LOOKM_TRY(check_workspace(pl, workspace, workspace_bytes));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    LOOKM_TRY(begin_call(pl, workspace, st));
    LOOKM_CUDA(launch_argmax_rows(sim_matrix, req_table(pl, workspace), pl.n_kv_heads,
                                  pl.max_E, assign, sim, st));
    ++g_launches;
    return LOOKM_OK;
}

int lookm_merge(const void* k, const void* v, const int* kept_idx, const int* evict_idx,
                const int* assign, const float* sim, const int* cu_seqlens_host, int n_requests,
                const int* budgets_host, const int* merge_modes_host, const lookm_layout* layout,
                int varlen_output, void* out_k, void* out_v, void* workspace,
                size_t workspace_bytes, void* cuda_stream) {
    if (!k || !v || !kept_idx || !evict_idx || !cu_seqlens_host || !budgets_host || !merge_modes_host ||
        !out_k || !out_v)
        return LOOKM_ERR_INVALID_ARG;
    if (!varlen_output && n_requests != 1) return LOOKM_ERR_INVALID_ARG;
    Plan pl;
    LOOKM_TRY(build_plan(pl, layout, n_requests, cu_seqlens_host, nullptr, budgets_host, nullptr,
                         merge_modes_host));
    if ((!assign || !sim) && pl.n_none < pl.n_req) return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_layout_ptrs(layout, nullptr, k, v));
    LOOKM_TRY(check_out_ptrs(out_k, out_v));
    LOOKM_TRY(check_word_ptrs({kept_idx, evict_idx, assign, sim}));
    LOOKM_TRY(set_out_stride(pl, varlen_output, 0));
    LOOKM_TRY(check_workspace(pl, workspace, workspace_bytes));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    LOOKM_TRY(begin_call(pl, workspace, st));
    return run_merge(pl, layout, k, v, kept_idx, evict_idx, assign, sim, varlen_output, out_k, out_v,
                     workspace, st);
}

int lookm_device_status(void* workspace, void* cuda_stream) {
    if (!workspace) return LOOKM_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int word = 0;
    if (cudaStreamSynchronize(st) != cudaSuccess) return LOOKM_ERR_CUDA;
    if (cudaMemcpy(&word, workspace, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return LOOKM_ERR_CUDA;
    if (word != 0 && cudaMemset(workspace, 0, sizeof(int)) != cudaSuccess) return LOOKM_ERR_CUDA;
    return word;
}

int lookm_selftest_wait_expiry(int limit_us, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (limit_us < 1 || limit_us > 100000) return LOOKM_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return LOOKM_ERR_INVALID_ARG;
    if (workspace_bytes < 256) return LOOKM_ERR_WORKSPACE_TOO_SMALL;
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    g_launches = 0;
    LOOKM_CUDA(cudaMemsetAsync(workspace, 0, 256, st));
    LOOKM_CUDA(launch_wait_probe(1000ull * (unsigned long long)limit_us, static_cast<int*>(workspace), st));
    ++g_launches;
    return LOOKM_OK;
}

int lookm_last_launch_count(void) { return g_launches; }

int lookm_set_stage_events(void* const* events_host, int n_events) {
    if (!events_host || n_events == 0) { g_stage_events = nullptr; return LOOKM_OK; }
    if (n_events != LOOKM_N_STAGE_EVENTS) return LOOKM_ERR_INVALID_ARG;
    g_stage_events = events_host;
    return LOOKM_OK;
}

const char* lookm_strerror(int status) {
    switch (status) {
        case LOOKM_OK: return "ok";
        case LOOKM_ERR_INVALID_ARG: return "invalid argument";
        case LOOKM_ERR_UNSUPPORTED: return "unsupported configuration or device";
        case LOOKM_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case LOOKM_ERR_CUDA: return "a CUDA call failed";
        case LOOKM_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait expired";
        case LOOKM_ERR_DEVICE_BAD_INDEX: return "an index list held an out-of-range entry";
        default: return "unknown status";
    }
}

}  // extern "C"

// ------------------------------------------------------------------------------------------------
// lookm_merge_noalloc: the merge step with its scratch in a static device array.
// ------------------------------------------------------------------------------------------------
namespace {

// Scratch of the no-allocation merge: status word, request table, entry lists, per-slot counters,
// per-unit records and the two sort buffers.  Lives in the library's device image, so every GPU that loads the library holds
// these bytes until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[LOOKM_NOALLOC_SCRATCH_BYTES];

// Device address of the array on the current device.  The array's name is only a host-side
// handle here; kernels must be given the address cudaGetSymbolAddress returns.  Looked up once
// per device (with that device current) and cached.
int noalloc_scratch_ptr(void** out) {
    static std::mutex mu;
    static void* cache[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LOOKM_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!cache[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return LOOKM_ERR_CUDA;
        cache[dev] = p;
    }
    *out = cache[dev];
    return LOOKM_OK;
}

}  // namespace

extern "C" int lookm_merge_noalloc(const void* k, const void* v, const int* kept_idx,
                                   const int* evict_idx, const int* assign, const float* sim,
                                   const int* cu_seqlens_host, int n_requests,
                                   const int* budgets_host, const int* merge_modes_host,
                                   const lookm_layout* layout, int varlen_output, void* out_k,
                                   void* out_v, void* cuda_stream) {
    if (!k || !v || !kept_idx || !evict_idx || !assign || !sim || !cu_seqlens_host || !budgets_host ||
        !merge_modes_host || !out_k || !out_v)
        return LOOKM_ERR_INVALID_ARG;
    if (!varlen_output && n_requests != 1) return LOOKM_ERR_INVALID_ARG;
    Plan pl;
    LOOKM_TRY(build_plan(pl, layout, n_requests, cu_seqlens_host, nullptr, budgets_host, nullptr,
                         merge_modes_host));
    LOOKM_TRY(check_layout_ptrs(layout, nullptr, k, v));
    LOOKM_TRY(check_out_ptrs(out_k, out_v));
    LOOKM_TRY(check_word_ptrs({kept_idx, evict_idx, assign, sim}));
    LOOKM_TRY(set_out_stride(pl, varlen_output, 0));
    // compact carving of just what the merge needs: 28 bytes per (KV head, token), 4 per kept row,
    // the per-unit records and the table
    const size_t units = (size_t)pl.n_kv_heads * (size_t)pl.T;
    size_t o = 0;
    auto carve = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    pl.clear_words = 64;
    pl.o_status = carve(256);
    pl.o_reqs = carve(sizeof(Req) * (size_t)n_requests);
    pl.o_row_begin = carve(4 * (units + (size_t)pl.n_kv_heads * (size_t)n_requests));
    pl.o_entries = carve(8 * units);
    pl.o_units = carve(16 * (size_t)pl.total_units);
    pl.o_slot_cnt = carve(4 * (size_t)pl.total_slots);
    pl.o_parts = carve((size_t)kMergePartBytes * (size_t)pl.total_units);
    pl.o_sort_a = carve(8 * units);
    pl.o_sort_b = carve(8 * units);
    pl.total = o;
    if (pl.total > (size_t)LOOKM_NOALLOC_SCRATCH_BYTES) return LOOKM_ERR_WORKSPACE_TOO_SMALL;
    void* scratch = nullptr;
    LOOKM_TRY(noalloc_scratch_ptr(&scratch));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // begin_call clears the status word and rewrites the table; every list the kernels read is
    // rewritten by the inversion kernel first, so nothing else of the last call's contents matters.
    LOOKM_TRY(begin_call(pl, scratch, st));
    return run_merge(pl, layout, k, v, kept_idx, evict_idx, assign, sim, varlen_output, out_k, out_v,
                     scratch, st);
}

extern "C" int lookm_noalloc_status(void* cuda_stream) {
    void* scratch = nullptr;
    LOOKM_TRY(noalloc_scratch_ptr(&scratch));
    return lookm_device_status(scratch, cuda_stream);
}

// ------------------------------------------------------------------------------------------------
// Generation step over a cache (Section 3.1, Eq. 2-3): host planner of decode_kernel.cu.
// ------------------------------------------------------------------------------------------------
namespace {

constexpr int kDecodeClusterRows = 256;
constexpr int kDecodeStepRows = 64;         // rows a CTA of any decode kernel takes at a time

// One way to take the step: which kernel, and how the caches are cut.
struct DecodeWay {
    int gt = 1, n_pass = 1;                 // query heads per pass over the rows, passes per group
    bool mma = false;
    long long rows_per_split = 64;
    int cluster = 1;                        // > 1: so many splits everywhere, added up inside the launch
    bool shares = false;                    // the CTAs take equal shares of all rows (one query head at a time)
    double us = 0.;                         // estimated time
};
struct DecodePlan {
    int n_req = 0;
    DecodeWay way;
    std::vector<DecodeReq> reqs;            // caller order
    size_t o_parts = 0, total = 0;
};

int decode_sms() {
    DeviceInfo di;
    return (device_info(di) == LOOKM_OK && di.sms > 0) ? di.sms : 148;
}

// Time of a step in us: a launch, the CTAs' steps of 64 rows in every wave of CTAs, a start per further
// wave, and where the splits take a second launch that and its chain over the splits.  Fitted to 400 steps
// (groups of 2 to 16 heads, 1 to 32 KV heads, 1 to 32768 rows, 1 to 100 requests); the way it picks takes 0.5 %
// longer than the fastest of the three on average and 10 % at most.
struct DecodeCost { double launch, step, wave, combine, splits16; };
constexpr DecodeCost kCostOneHead = {0.9, 0.59, 1.0, 2.4, 0.7}, kCostTwoHeads = {1.25, 0.78, 1.4, 2.6, 0.7},
                     kCostMma = {1.9, 1.33, 1.35, 2.7, 0.85};
constexpr double kMmaStepAlone = 1.9;       // of a CTA that has its SM to itself and waits for each of its steps

// Most rows that an SM gets when whole splits (of s rows at most) go in order to whichever of `wave` SMs is free
// first: SMs with the same load, as (load, how many), move on together.
long long most_rows(const int* lens, int n_req, long long units, long long s, long long wave) {
    typedef std::pair<long long, long long> Load;
    std::vector<Load> room;
    room.reserve(128);
    std::priority_queue<Load, std::vector<Load>, std::greater<Load>> free(std::greater<Load>(), std::move(room));
    free.push({0, wave});
    long long most = 0;
    const auto give = [&](long long rows, long long pieces) {
        while (pieces > 0) {
            Load l = free.top();
            free.pop();
            const long long n = std::min(pieces, l.second);
            if (l.second > n) free.push({l.first, l.second - n});
            free.push({l.first + rows, n});
            most = std::max(most, l.first + rows);
            pieces -= n;
        }
    };
    for (int r = 0; r < n_req; ++r) {
        const long long rows = (long long)lens[r] + 1;
        give(std::min(s, rows), units * ((rows + s - 1) / s));
    }
    return most;
}

// Time of the slowest CTA of each launch in equal shares: so much per step of 64 rows, while two CTAs work on an SM, per
// unit, and per further launch.  A share has most units where it begins with a request or ends with one (the shares lie where
// they lie: this is up to a unit off); the walk costs 0.1 us per eight requests, one over the CTAs' shares 1 to 2 us.
constexpr double kShareStepUs = 1.3, kShareUnitUs = 0.86, kShareLaunchUs = 4.2;
double slowest_share(const int* lens, int n_req, long long units, int sms) {
    double us = -kShareLaunchUs;
    for (int base = 0; base < n_req; base += kDecodeChunk) {
        const int n = std::min(kDecodeChunk, n_req - base);
        long long per[kDecodeChunk], steps = 0;                       // steps of a unit
        for (int r = 0; r < n; ++r) {
            per[r] = lens[base + r] / kDecodeShareRows + 1;
            steps += per[r] * units;
        }
        const long long ctas = std::min<long long>((long long)sms * kDecodeShareCtasPerSm, steps), share = (steps + ctas - 1) / ctas;
        long long most = 1;
        for (int step : {1, -1})
            for (int from = 0; from < n; ++from) {
                if (from > 0 && from < n - 1 && per[from] >= per[from - step]) continue;          // (denser units lie before it)
                long long left = share, count = 0;
                for (int r = from; r >= 0 && r < n && left > 0; r += step) {
                    const long long here = std::min(left, per[r] * units);
                    count += here == left ? (here + per[r] - 1) / per[r] : units;
                    left -= here;
                }
                most = std::max(most, count);
            }
        us += kShareLaunchUs + (double)share * kShareStepUs + (double)most * kShareUnitUs;
    }
    return us;
}

DecodeWay decode_way(const lookm_cache_layout* lay, int n_req, const int* lens, int gt, bool mma, int sms) {
    DecodeWay w;
    w.gt = gt;
    w.mma = mma;
    w.n_pass = lay->n_q_heads / lay->n_kv_heads / gt;
    const long long units = (long long)lay->n_kv_heads * w.n_pass;       // (KV head, pass) per request
    // The grid is one wave: as many CTAs as the GPU holds at a time (a second, partly filled wave
    // would cost as much as the first).  Rows per split: the smallest count with which the splits
    // of all requests fit into that wave; on the tensor cores, where a short step takes as long as a
    // full one, two steps at least.
    const int per_sm = decode_ctas_per_sm(gt, mma);
    const long long wave = (long long)sms * (per_sm > 0 ? per_sm : 2);
    long long total_rows = 0;
    int longest = 0;
    for (int r = 0; r < n_req; ++r) {
        total_rows += ((long long)lens[r] + 1) * units;
        longest = std::max(longest, lens[r] + 1);
    }
    auto ctas_with = [&](long long rows) {
        long long c = 0;
        for (int r = 0; r < n_req; ++r) c += (((long long)lens[r] + rows) / rows) * units;
        return c;
    };
    long long s = std::max<long long>(mma ? 2 * kDecodeStepRows : 16, (total_rows + wave - 1) / wave);
    if (ctas_with(s) > wave) {
        // smallest count in (s, longest cache + 1] that fits (the CTA count never grows with
        // it); with the upper end every request is a single split, the least there can be
        long long lo = s, hi = std::max<long long>(s, longest);
        while (lo < hi) {
            const long long mid = lo + (hi - lo) / 2;
            if (ctas_with(mid) > wave) lo = mid + 1; else hi = mid;
        }
        s = lo;
    }
    // 2, 4 or 8 splits per (KV head, pass) that one cluster adds up, instead of a second launch: as
    // many as leave every CTA an SM of its own (clusters of 8 fill about two thirds of the SMs
    // before two share one, smaller ones seven eighths: 16 heads x 8 took 5.7 us where 12 x 8 took
    // 3.1).  Worth it while a split is short, or at any length if the CTAs cover nearly all SMs (one
    // request of 32 heads x 4 or 64 x 2: 119 to 129 CTAs);
    // us per step, two launches | one: 32 heads x 4 splits 409 rows 4.6 | 3.8, 3000 rows 10.2 | 9.2, 32768 rows
    // 78.9 | 79.9; 31 x 4 8192 rows 23.3 | 22.1; 60 x 2 8192 rows 41.2 | 39.8; 64 x 2 32768 rows 165 | 159; 12 x 8
    // 1638 rows 5.3 | 4.9, 8192 rows 12.6 | 13.0; 16 x 4 800 rows 4.6 | 4.7 (8.0 | 5.8 with the launches issued one
    // by one), 3000 rows 6.9 | 9.0.
    int c = kDecodeMaxCluster;
    while (c > 1 && n_req * units * c > (c == 8 ? sms * 2 / 3 : sms * 7 / 8)) c /= 2;
    const long long rows = (longest + c - 1) / c;
    if (c > 1 && s < longest && (rows <= kDecodeClusterRows || (n_req == 1 && units * c >= sms * 4 / 5))) {
        w.cluster = c;
        s = rows;
    }
    w.rows_per_split = s;
    const long long ctas = w.cluster > 1 ? n_req * units * w.cluster : ctas_with(s), splits = (longest + s - 1) / s;
    const double waves = (double)std::max<long long>(1, (ctas + wave - 1) / wave);
    const double steps = (double)((std::min<long long>(s, longest) + kDecodeStepRows - 1) / kDecodeStepRows);
    const DecodeCost& cost = mma ? kCostMma : gt == 2 ? kCostTwoHeads : kCostOneHead;
    w.us = cost.launch + waves * steps * (mma && ctas <= sms ? kMmaStepAlone : cost.step) + (waves - 1.) * cost.wave;
    if (w.cluster == 1 && splits > 1) w.us += cost.combine + cost.splits16 * std::max<long long>(0, splits - 16) / 16.;
    if (gt == 1 && !mma) {
        // Equal shares?  Whole splits take as long as memory needs for all rows, or as long as an SM needs for the
        // most rows that it gets, with a start per further wave and mostly a second launch.  Shares, nearly always two launches,
        // take as long as the CTA whose steps and units together take longest: a share of many short units lasts longer
        // than the others.  Fitted to 350 steps of 1 to 150 requests, 10 to 32768 rows and 1 to 100 heads, both ways; from 8 us on
        // the estimates are 5 % off.  Of 1200 steps that follow this rule, half of them in shares, one in shares takes 8 %
        // longer than in whole splits and seven 3 to 5.  us, whole | shares: 4 requests of 1000 to 8000 rows x 32 heads 76 | 47,
        // 14 of 2000 to 6000 x 8 47.6 | 38.9, 64 of 40 x 32 38 | 18, one of 32768 x 40 117 | 108; left whole: nine of 61 to
        // 4390 x 32, the 61 in one share, 60.7 | 86.5, 33 of 54 to 1168 x 8 18.3 | 21.3, 36 of 22 to 1088 x 16 34.7 | 43.4, one of
        // 8990 x 16 15.1 | 17.1.
        constexpr double kRowUs = 7.9e-5, kSmRowUs = 9.6e-3, kStartUs = 2.8, kWaveUs = 2.1, kCombineUs = 1.3, kShareUs = 3.7,
                         kLaunchUs = 0.5;
        const bool combined = w.cluster == 1 && splits > 1;
        // (the heads of a group find their rows in L2)
        const double from_memory = (double)total_rows / (double)w.n_pass * kRowUs, later_waves = std::max(0., (double)ctas / (double)wave - 1.);
        const auto whole_with = [&](double most) {
            return std::max(most * kSmRowUs + later_waves * kWaveUs, from_memory) + kStartUs + (combined ? kCombineUs : 0.);
        };
        // The most rows of an SM are no fewer than the mean and a split's, and no more than both together; worked out only where
        // that leaves it open.  (A launch more also takes the host longer.)
        const double mean = (double)total_rows / (double)wave, piece = (double)std::min<long long>(s, longest);
        double whole = whole_with(ctas <= wave ? piece : std::max(mean, piece));
        const double slower = ctas <= wave ? whole : whole_with(mean + piece);
        if (slower > kShareUs + kShareStepUs + kShareUnitUs) {               // (no share is shorter)
            const double shares = std::max(slowest_share(lens, n_req, units, sms), from_memory) + kShareUs +
                                  (!combined && longest > kDecodeShareRows ? kLaunchUs : 0.);
            const auto pays = [&](double whole) { return shares + std::min(0.06 * whole, 1.6) < whole; };
            if (!pays(whole) && pays(slower)) whole = whole_with((double)most_rows(lens, n_req, units, s, wave));
            w.shares = pays(whole);
            if (w.shares) w.us += shares - whole;
        }
        if (w.shares) w.cluster = 1;
    }
    return w;
}

// lens may be NULL (sizing only).  The workspace is sized for the largest number of splits any
// lengths can produce, so a cache may grow from step to step under one workspace.
int build_decode_plan(DecodePlan& dp, const lookm_cache_layout* lay, int n_req, const long long* begins,
                      const int* lens) {
    if (!lay || n_req <= 0) return LOOKM_ERR_INVALID_ARG;
    if (lay->head_dim != kHeadDim) return LOOKM_ERR_UNSUPPORTED;
    if (lay->n_kv_heads <= 0 || lay->n_q_heads <= 0 || lay->n_q_heads % lay->n_kv_heads)
        return LOOKM_ERR_INVALID_ARG;
    if (lay->n_q_heads > 65535 || n_req > (1 << 20)) return LOOKM_ERR_UNSUPPORTED;
    if (lay->cache_stride_row <= 0 || lay->cache_stride_head <= 0 || lay->cache_stride_row % 8 ||
        lay->cache_stride_head % 8)
        return LOOKM_ERR_INVALID_ARG;
    if (!(lay->softmax_scale >= 0.f) || !std::isfinite(lay->softmax_scale)) return LOOKM_ERR_INVALID_ARG;
    const int group = lay->n_q_heads / lay->n_kv_heads;
    dp.n_req = n_req;
    int widest = std::min(group, 8);        // largest divisor of the group up to 8
    while (group % widest) --widest;
    const int sms = decode_sms();
    if (lens) {
        for (int r = 0; r < n_req; ++r)
            if (lens[r] < 0 || lens[r] >= (1 << 30) || (begins && begins[r] < 0)) return LOOKM_ERR_INVALID_ARG;
        // Query heads of a group one by one, two by two, or all of them on the tensor cores.  Which is the
        // fastest depends on the rows, the heads and the requests together, us: 32 heads on 16 with 409 rows
        // 3.7, 4.0 and 5.5, with 3276 9.7, 8.8 and 9.4, with 32768 74, 50 and 45; 64 requests of 30 rows, 16 heads
        // on 1, 13.4, 9.5 and 4.4; 32 heads on 8 with 409 rows 3.7, 4.0 and 4.3, with 8192 20.6, 16.0 and 11.4.
        dp.way = decode_way(lay, n_req, lens, 1, false, sms);
        if (group > 1) {
            // (shares of single heads by a clear margin only: of one cache of 28811 rows, 96 heads on 32, 184 us estimated
            // against 217 on the tensor cores were 165 against 160)
            const auto better = [&](const DecodeWay& w) { if (w.us < (dp.way.shares ? 1.25 : 1.) * dp.way.us) dp.way = w; };
            if (group % 2 == 0) better(decode_way(lay, n_req, lens, 2, false, sms));
            if (widest > 1) better(decode_way(lay, n_req, lens, widest, true, sms));
        }
        if (dp.way.rows_per_split >= (1ll << 31)) return LOOKM_ERR_UNSUPPORTED;
    }
    // at most one wave of the fullest kernel, or one (short) split per (request, KV head, pass)
    // when the batch alone has more units than a wave holds; with the most heads per pass these
    // records need the most room
    const long long units = (long long)lay->n_kv_heads * (group / widest);
    const long long max_splits = (long long)kDecodeMaxCtasPerSm * sms + (long long)n_req * units;
    if (max_splits * widest >= (1ll << 31)) return LOOKM_ERR_UNSUPPORTED;
    if (lens) {
        dp.reqs.resize(n_req);
        long long parts = 0;
        const long long s = dp.way.rows_per_split;
        for (int r = 0; r < n_req; ++r) {
            DecodeReq& q = dp.reqs[r];
            q.begin = begins ? begins[r] : 0;
            q.len = lens[r];
            q.index = r;
            q.n_splits = dp.way.cluster > 1 ? dp.way.cluster : (int)(((long long)lens[r] + 1 + s - 1) / s);
            q.cta_begin = 0;
            q.part_begin = parts;
            parts += (long long)q.n_splits * lay->n_kv_heads * dp.way.n_pass * dp.way.gt;
        }
    }
    size_t o = 0;
    auto carve = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    dp.o_parts = carve(4 * (size_t)(kHeadDim + 2) * (size_t)max_splits * (size_t)widest);
    dp.total = o;
    return LOOKM_OK;
}

int decode_common(const void* q, const void* k_new, const void* v_new, void* cache_k, void* cache_v,
                  const long long* begins, const int* lens, int n_req, const lookm_cache_layout* lay,
                  float* out, void* ws, size_t ws_bytes, void* stream) {
    if (!q || !k_new || !v_new || !cache_k || !cache_v || !lens || !out) return LOOKM_ERR_INVALID_ARG;
    for (const void* p : {q, k_new, v_new, (const void*)cache_k, (const void*)cache_v})
        if (reinterpret_cast<uintptr_t>(p) & 15u) return LOOKM_ERR_INVALID_ARG;
    LOOKM_TRY(check_word_ptrs({out}));
    DecodePlan dp;
    LOOKM_TRY(build_decode_plan(dp, lay, n_req, begins, lens));
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u)) return LOOKM_ERR_INVALID_ARG;
    if (ws_bytes < dp.total) return LOOKM_ERR_WORKSPACE_TOO_SMALL;
    DeviceInfo di;
    LOOKM_TRY(device_info(di));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    g_launches = 0;
    const float scale = lay->softmax_scale > 0.f ? lay->softmax_scale : 1.0f / std::sqrt((float)lay->head_dim);
    const long long units = (long long)lay->n_kv_heads * dp.way.n_pass;
    for (int base = 0; base < n_req; base += kDecodeChunk) {
        DecodeBatch batch;
        std::memset(&batch, 0, sizeof(batch));
        batch.n_req = std::min(kDecodeChunk, n_req - base);
        long long ctas = 0, steps = 0;
        bool split = false;
        for (int i = 0; i < batch.n_req; ++i) {
            batch.r[i] = dp.reqs[base + i];
            batch.r[i].cta_begin = (int)ctas;
            ctas += (long long)batch.r[i].n_splits * units;
            split = split || (batch.r[i].n_splits > 1 && dp.way.cluster == 1);
            if (dp.way.shares) {
                const int unit = batch.r[i].len / kDecodeShareRows + 1;
                batch.r[i].step_begin = steps;
                steps += unit * units;
                split = split || unit > 1;
            }
        }
        if (dp.way.shares) {
            ctas = std::min<long long>((long long)di.sms * kDecodeShareCtasPerSm, steps);
            if (steps / ctas >= (1ll << 30)) return LOOKM_ERR_UNSUPPORTED;
            batch.share = (int)(steps / ctas);
            batch.longer = (int)(steps % ctas);
        }
        if (ctas >= (1ll << 31)) return LOOKM_ERR_UNSUPPORTED;
        LOOKM_CUDA(launch_decode(batch, (int)ctas, dp.way.gt, dp.way.mma, dp.way.cluster, q, k_new, v_new, cache_k, cache_v,
                                 lay->cache_stride_row, lay->cache_stride_head, lay->n_q_heads,
                                 lay->n_kv_heads, (int)dp.way.rows_per_split, scale * 1.4426950408889634f,
                                 at<float>(ws, dp.o_parts), out, st));
        ++g_launches;
        if (split) {
            LOOKM_CUDA(launch_decode_combine(batch, dp.way.gt, lay->n_q_heads, lay->n_kv_heads,
                                             scale * 1.4426950408889634f, at<float>(ws, dp.o_parts), out, st));
            ++g_launches;
        }
    }
    return LOOKM_OK;
}

}  // namespace

extern "C" size_t lookm_decode_workspace_size(const lookm_cache_layout* layout, int n_requests,
                                              const int* cache_lens_host) {
    DecodePlan dp;
    if (build_decode_plan(dp, layout, n_requests, nullptr, cache_lens_host) != LOOKM_OK) return 0;
    return dp.total;
}

extern "C" int lookm_decode_step(const void* q, const void* k_new, const void* v_new, void* cache_k,
                                 void* cache_v, int cache_len, const lookm_cache_layout* layout,
                                 float* out, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    const long long begin = 0;
    return decode_common(q, k_new, v_new, cache_k, cache_v, &begin, &cache_len, 1, layout, out, workspace,
                         workspace_bytes, cuda_stream);
}

extern "C" int lookm_decode_step_varlen(const void* q, const void* k_new, const void* v_new, void* cache_k,
                                        void* cache_v, const long long* cache_begin_host,
                                        const int* cache_lens_host, int n_requests,
                                        const lookm_cache_layout* layout, float* out, void* workspace,
                                        size_t workspace_bytes, void* cuda_stream) {
    if (!cache_begin_host) return LOOKM_ERR_INVALID_ARG;
    return decode_common(q, k_new, v_new, cache_k, cache_v, cache_begin_host, cache_lens_host, n_requests,
                         layout, out, workspace, workspace_bytes, cuda_stream);
}
