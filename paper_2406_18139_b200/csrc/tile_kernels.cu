// The two sweeps of the cumulative attention score (Eq. 4).
//
// Both are the same persistent, warp-specialised pipeline over 128 x 128 x 128 bf16 tiles:
//   - a work item owns one STATIONARY 128-row tile (the A operand, rows on the 128 TMEM lanes)
//     and streams a sequence of 128-row tiles (the B operand) against it;
//   - warp 0 (one thread) issues the TMA loads, warps 1 and 18 (one thread each, tiles taken
//     alternately) issue tcgen05.mma into one of four 128-column TMEM accumulators, and four
//     groups of four warps read the accumulators with tcgen05.ld and run the epilogue; group w
//     owns accumulator w and takes the tiles whose running index is w mod 4, so each SM
//     sub-partition always has four epilogue warps to switch between;
//   - each epilogue thread owns one row of the stationary tile, so every reduction over the
//     streamed axis (row maximum and sum, column-sum of probabilities for one key) stays in
//     that thread's registers; the four groups are combined through shared memory once per
//     item.  No L x L matrix is ever stored.
//
//   sweep 1: A = 128 queries of one query head, B = key tiles 0..diagonal.  Online softmax
//            statistics per query row  ->  lse[i] = log sum_{j<=i} exp(s_ij).
//   sweep 2: A = 128 keys of one KV head, B = query tiles diagonal..last of every query head in
//            the group.  Thread of key j accumulates sum_i exp(s_ij - lse_i)  ->  A_s[j].  The
//            subtraction of lse_i is done by the tensor core: sweep 1 leaves -lse_i / scale as
//            three bf16 terms in a 16-column companion of the query tensor, and a ninth MMA per
//            tile multiplies it with a constant tile of ones, so the accumulator already holds
//            s_ij - lse_i / scale and the epilogue needs no per-column data at all.
//
// A small problem has fewer or more uneven sweep items than the CTAs can share.  Then the streamed tiles of an item are cut into
// p.splits ranges, items of their own that leave partial results in memory; the one that arrives last
// (a counter per 32 rows) adds them in range order.  Large problems run a kernel without that code (with
// it 8192 tokens x 32 heads took 1.5 % longer).
//
// Work items are laid out heaviest first and dealt to the CTAs in serpentine order; every role
// walks the same item sequence on its own, so no scheduling state is shared.
#include <cuda_bf16.h>
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace lookm {
namespace {

#ifndef LOOKM_TILE_STAGES
#define LOOKM_TILE_STAGES 4
#endif
#ifndef LOOKM_TILE_ABUF
#define LOOKM_TILE_ABUF 2
#endif
constexpr int kStages = LOOKM_TILE_STAGES;       // ring of streamed tiles
constexpr int kABuf = LOOKM_TILE_ABUF;           // buffers of the stationary tile (2: the next item's is
                                                 // loaded while this item's is in use)
constexpr int kAccum = 4;                        // TMEM accumulators (128 fp32 columns each)
constexpr int kGroups = 4;                       // epilogue groups of four warps; tile g goes to group g mod kGroups
// "Accumulator filled" barriers form a ring twice as long as the accumulators: tile g uses barrier
// g mod kFullRing in phase g / kFullRing.  A group may reach tile g while tile g - kAccum (same
// accumulator, other group, other issuing thread) is still being multiplied; with one barrier per
// accumulator its parity wait would then pass at once.  With the longer ring the tile one phase
// back is g - 2 kAccum, whose MMAs had to complete before the producer could load tile g - kAccum,
// which it did before it loaded any tile this group has already finished.
constexpr int kFullRing = 2 * kAccum;
constexpr int kIssuers = 2;                      // MMA-issuing threads (tiles alternate between them)
constexpr int kEpiWarp0 = 2;                     // first epilogue warp
// producer warp, MMA warp, kGroups x 4 epilogue warps, second MMA warp
constexpr int kThreads = 64 + kGroups * 128 + 32;
constexpr int kHalfBytes = kTile * 64 * 2;       // one TMA box: 128 rows x 64 bf16 (128 B rows)
constexpr int kTileBytes = 2 * kHalfBytes;       // 128 x 128 bf16
constexpr int kSplitBytes = kTile * 16 * 2;      // 128 rows x 16 bf16 (32-byte rows, 32-byte swizzle)
constexpr int kItemRing = 4;                     // items announced to the roles of a CTA (multi_kernel)
constexpr int kReqCache = 16;                    // request-table entries cached in shared memory
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kReferenceSlack = 1.152921504606847e18f;   // 2^60: largest chunk sum kept against a stale reference
constexpr float kReferenceSlackLog2 = 60.f;
constexpr float kLn2 = 0.6931471805599453f;

template <int KIND>
struct __align__(1024) Shared {
    static constexpr int kXStages = (KIND == kSweep2) ? kStages : 1;   // only sweep 2 streams companions
    static constexpr int kPlanes = (KIND == kSweep2) ? 1 : 2;          // values per row and group to combine
    uint8_t a[kABuf][kTileBytes];                // stationary tiles
    uint8_t b[kStages][kTileBytes];              // streamed tiles
    uint8_t bx[kXStages][kSplitBytes];           // sweep 2: the streamed tiles' 16-column companions
    uint8_t ax[kSplitBytes];                     // sweep 2: constant ones tile that multiplies bx
    float comb[2][kGroups][kPlanes][kTile];       // partial results of the groups, double-buffered
    Req reqs[kReqCache];                         // copy of the request table (when it fits)
    unsigned long long a_full[kABuf], a_empty[kABuf];
    unsigned long long b_full[kStages], b_empty[kStages];
    unsigned long long t_full[2 * kAccum], t_empty[kAccum];   // t_full: see kFullRing
    unsigned long long comb_full[2], comb_free[2];   // partial results of an item written / read
    unsigned long long mma_done;                 // every MMA of this CTA has completed
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(Shared<kSweep1>) + 1024 <= 232448 && sizeof(Shared<kSweep2>) + 1024 <= 232448,
              "shared memory of the tile kernels exceeds 227 KB");

// The softmax epilogues are bound by the special-function unit (16 ex2 per clock and SM) and by issue
// slots, so some columns are exponentiated on the FMA pipe instead: on full tiles kPolyPairs of the sixteen pairs
// of a chunk, two numbers per instruction, with one test of the largest logit (of a chunk in sweep 1, of a whole item in
// sweep 2) in place of an upper limit on every argument (which took two instructions a pair more).  A two-wide multiply-add takes two issue
// slots, so it is the limit's instructions that are saved.  Scores in us, one column in six one by one | 2, 3, 5, 6 and 7
// pairs: 8192 tokens x 32 heads 678 | 676, 669, 684, 700, 726; 4096 x 32 191.3 | 189.4, 190.4, 195.9, 202.8, 210.5; three
// prompts of 1800 to 5000 x 32 on 8 552 | 549, 548, 567, 583, 605.
constexpr int kPolyPairs = 3;
__host__ __device__ constexpr bool poly_pair(int i) { return ((i + 1) * kPolyPairs) / 16 != (i * kPolyPairs) / 16; }
__device__ __forceinline__ ptx::f32x2 exp2_pair(int i, ptx::f32x2 x) {
    if (poly_pair(i)) return ptx::ex2_fma2(x);
    const float2 v = ptx::unpack2(x);
    return ptx::pack2(ptx::ex2(v.x), ptx::ex2(v.y));
}
// Diagonal tiles: one column in kPolyEvery.
constexpr int kPolyEvery = 6;
__device__ __forceinline__ float exp2_mixed(int column, float x) {
    return (column % kPolyEvery == kPolyEvery - 1) ? ptx::ex2_fma(x) : ptx::ex2(x);
}

// ---- epilogue of the sweeps on 32 accumulator columns, one row per thread ------------------------
// Sweep 1: softmax statistics of a query row; l is the sum of exp2(x - m c2), where m is a REFERENCE,
// not necessarily the maximum so far.  Diagonal tile (the last of the item; columns from c0 on, usable
// up to `row`): exact running maximum.
__device__ __forceinline__ void sweep1_diagonal(const uint32_t (&raw)[32], int c0, int row, float c2, float& m, float& l) {
    float mx = m;
#pragma unroll
    for (int c = 0; c < 32; ++c)
        if (c0 + c <= row) mx = fmaxf(mx, __uint_as_float(raw[c]));
    if (mx != -INFINITY) {                               // false only above the diagonal
        const float mc = mx * c2;
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
            const float e0 = exp2_mixed(c, fmaf(__uint_as_float(raw[c]), c2, -mc));
            const float e1 = exp2_mixed(c + 1, fmaf(__uint_as_float(raw[c + 1]), c2, -mc));
            s0 += (c0 + c <= row) ? e0 : 0.f;
            s1 += (c0 + c + 1 <= row) ? e1 : 0.f;
        }
        l = l * ptx::ex2(m * c2 - mc) + (s0 + s1);
        m = mx;
    }
}
// Full tiles: no maximum is taken.  The reference is the maximum of the row's first 32 columns; later
// logits may exceed it as long as the chunk's sum stays below 2^60 (fp32 has the range, and the relative
// precision does not depend on the reference).  When it does not, or overflows, the chunk is redone
// against its true maximum.
__device__ __forceinline__ void sweep1_columns(const uint32_t (&raw)[32], float c2, float& m, float& l) {
    float ref = m;                                       // -inf at the row's first chunk: the sum
    float sum;                                           // overflows and the second round sets it
#pragma unroll 1
    for (int round2 = 0;; ++round2) {
        const float mc = ref * c2;
        const ptx::f32x2 scale = ptx::pack2(c2, c2), shift = ptx::pack2(-mc, -mc);
        ptx::f32x2 s[2] = {0ull, 0ull};
        float high = -INFINITY;                          // largest logit that the polynomial met, or NaN
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float a = __uint_as_float(raw[2 * i]), b = __uint_as_float(raw[2 * i + 1]);
            if (poly_pair(i)) high = ptx::fmax3_nan(high, a, b);
            s[i & 1] = ptx::add2(s[i & 1], exp2_pair(i, ptx::fma2(ptx::pack2(a, b), scale, shift)));
        }
        const float2 t = ptx::unpack2(ptx::add2(s[0], s[1]));
        sum = t.x + t.y;
        if ((sum < kReferenceSlack && fmaf(high, c2, -mc) < kReferenceSlackLog2) || round2) break;
        float mx = ref;
#pragma unroll
        for (int c = 0; c < 32; c += 2) mx = ptx::fmax3(mx, __uint_as_float(raw[c]), __uint_as_float(raw[c + 1]));
        l *= ptx::ex2(ref * c2 - mx * c2);
        if (!(high < INFINITY)) l = high - high;         // NaN, as the other unit makes it of such a logit
        ref = mx;
    }
    l += sum;
    m = ref;
}
// Sweep 2: probabilities of a key under 32 query columns (the accumulator holds s_ij - lse_i / scale);
// columns [from, limit) count.
__device__ __forceinline__ void sweep2_diagonal(const uint32_t (&raw)[32], int c0, int from, int limit, float c2, float (&acc)[4]) {
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        const float e = exp2_mixed(c, __uint_as_float(raw[c]) * c2);
        acc[c & 3] += (c0 + c >= from && c0 + c < limit) ? e : 0.f;
    }
}
// (high: the largest logit that the polynomial met, or NaN)
__device__ __forceinline__ void sweep2_columns(const uint32_t (&raw)[32], float c2, float (&acc)[4], float& high) {
    const ptx::f32x2 scale = ptx::pack2(c2, c2);
    ptx::f32x2 s[2] = {ptx::pack2(acc[0], acc[1]), ptx::pack2(acc[2], acc[3])};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float a = __uint_as_float(raw[2 * i]), b = __uint_as_float(raw[2 * i + 1]);
        if (poly_pair(i)) high = ptx::fmax3_nan(high, a, b);
        s[i & 1] = ptx::add2(s[i & 1], exp2_pair(i, ptx::mul2(ptx::pack2(a, b), scale)));
    }
    const float2 u = ptx::unpack2(s[0]), v = ptx::unpack2(s[1]);
    acc[0] = u.x;
    acc[1] = u.y;
    acc[2] = v.x;
    acc[3] = v.y;
}
// A row's sum, given the largest logit that the polynomial met: infinite from a probability of 2^128 on (a caller's
// log-sum-exp that is not one), of which the polynomial makes anything.
__device__ __forceinline__ float sweep2_sum(float sum, float high, float c2) {
    const float x = high * c2;
    return x < 128.f ? sum : x >= 128.f ? INFINITY : x;
}

// -lse / scale of one query row as three bf16 terms (their sum carries 24 bits) and 13 zeros:
// the row of the 16-column companion tensor that sweep 2 multiplies with ones.
__device__ __forceinline__ void store_lse_split(unsigned short* row16, float lse, float scale_log2) {
    const float u = -lse * (kLog2e / scale_log2);
    const __nv_bfloat16 hi = __float2bfloat16_rn(u);
    const float r1 = u - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    uint4 w0;
    w0.x = (uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(mid) << 16);
    w0.y = (uint32_t)__bfloat16_as_ushort(lo);
    w0.z = 0u;
    w0.w = 0u;
    uint4* dst = reinterpret_cast<uint4*>(row16);
    dst[0] = w0;
    dst[1] = make_uint4(0u, 0u, 0u, 0u);
}

// The single request of a call without a table writer, for the launches that read it from the table.
__device__ __forceinline__ void write_single_request(const ReqTable& reqs) {
    if (blockIdx.x == 0 && threadIdx.x < sizeof(Req) / 4)
        reinterpret_cast<int*>(const_cast<Req*>(reqs.rows))[threadIdx.x] = reinterpret_cast<const int*>(&reqs.only)[threadIdx.x];
}

__global__ void lse_split_kernel(const float* __restrict__ lse, int n_q_heads, long long T,
                                 float scale_log2, unsigned short* __restrict__ lse_split,
                                 const __grid_constant__ ReqTable reqs, int* clear, int n_clear) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // over [head][token]
    for (long long j = i; j < n_clear; j += (long long)gridDim.x * blockDim.x) clear[j] = 0;
    if (n_clear > 0) write_single_request(reqs);
    if (i >= T * n_q_heads) return;
    const long long h = i / T, tok = i % T;
    store_lse_split(lse_split + (tok * n_q_heads + h) * 16, lse[i], scale_log2);
}

// Row r of the ones tile: (1, 1, 1, 0, ... 0) in bf16; with the 32-byte swizzle the two 16-byte halves
// of a row trade places in rows 4-7 of every group of eight.
__device__ __forceinline__ void write_ones_row(uint8_t* ax, int r) {
    const int first = (r >> 2) & 1;
    uint4* row = reinterpret_cast<uint4*>(ax + r * 32);
    row[first] = make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
    row[first ^ 1] = make_uint4(0u, 0u, 0u, 0u);
    ptx::fence_proxy_async_shared();             // the tensor core reads it through the async proxy
}

struct Item {
    int tok_begin, L, blk, head, nt;
    int t0;                   // first streamed tile of the item (the sweeps' splits)
    int split, n_splits;      // which range of the block's tiles, of how many
    int tile;                 // index of the block over the whole batch
};

template <int KIND, bool kSplits, bool kOne>
__device__ __forceinline__ Item decode_item(const TileParams& p, const Req* tbl, int item) {
    int lo = 0, hi = kOne ? 0 : p.reqs.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tbl[mid].item_begin[KIND] <= item) lo = mid; else hi = mid - 1;
    }
    const Req& rq = tbl[lo];
    const int u = item - rq.item_begin[KIND];
    Item it;
    it.tok_begin = rq.tok_begin;
    it.L = rq.L;
    it.t0 = 0;
    it.split = 0;
    it.n_splits = 1;
    // heaviest first: last query block, first key block
    const int heads = (KIND == kSweep1 ? p.n_q_heads : p.n_kv_heads) * (kSplits ? p.splits : 1);
    const int b = u / heads, v = u % heads;
    it.blk = KIND == kSweep1 ? rq.nblk - 1 - b : b;
    it.nt = KIND == kSweep1 ? it.blk + 1 : (rq.nblk - it.blk) * p.group;
    it.head = v;
    if (kSplits) {
        it.head = v / p.splits;
        it.split = v % p.splits;
        it.n_splits = min(p.splits, it.nt);
        it.tile = rq.tile_begin + it.blk;
        const int all = it.nt;
        if (it.split < it.n_splits) {
            it.t0 = all * it.split / it.n_splits;
            it.nt = all * (it.split + 1) / it.n_splits - it.t0;
        } else {
            it.nt = 0;                           // no tile: every role passes over the item
        }
    }
    return it;
}

// Log-sum-exp of a query row (reference m in units of the accumulator, sum l) and its companion row.
__device__ __forceinline__ void store_lse(const TileParams& p, int head, int tok, float m, float l) {
    const float lse = (m * p.scale_log2 + ptx::lg2(l)) * kLn2;       // natural log, of the scaled logits
    p.lse[(long long)head * p.T + tok] = lse;
    store_lse_split(p.lse_split + ((long long)tok * p.n_q_heads + head) * 16, lse, p.scale_log2);
}

// Serpentine deal of the item list: round k hands items k*G .. k*G+G-1 to the CTAs in forward
// order when k is even and in reverse order when k is odd.
__device__ __forceinline__ int item_of_round(int round, int cta, int n_cta) {
    return round * n_cta + ((round & 1) ? (n_cta - 1 - cta) : cta);
}

// kOne: of a single request, which comes with the launch and may have no launch before it.  (Variants of their own: that code in
// the sweeps of batches cost 0.2 to 0.5 us a call, scores of four prompts of 134 to 1009 tokens x 16 heads 32.49 | 32.95.)
template <int KIND, bool kSplits, bool kOne>
__global__ void __launch_bounds__(kThreads, 1)
tile_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_x, const TileParams p) {
    extern __shared__ uint8_t smem_raw[];
    Shared<KIND>& sh = *reinterpret_cast<Shared<KIND>*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile int* abort_flag = &sh.abort_flag;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kABuf; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.a_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.a_empty[i]), kIssuers);
        }
        for (int i = 0; i < kStages; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.b_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.b_empty[i]), 1);
        }
        for (int i = 0; i < kFullRing; ++i) ptx::mbar_init(ptx::smem_u32(&sh.t_full[i]), 1);
        for (int i = 0; i < kAccum; ++i)
            ptx::mbar_init(ptx::smem_u32(&sh.t_empty[i]), 4);   // one arrival per epilogue warp of a group
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.comb_full[i]), (kGroups - 1) * 4);    // warps of the other groups
            ptx::mbar_init(ptx::smem_u32(&sh.comb_free[i]), 4);                   // warps of the combining group
        }
        ptx::mbar_init(ptx::smem_u32(&sh.mma_done), kIssuers);
        sh.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (KIND == kSweep2 && threadIdx.x < kTile) {
        write_ones_row(sh.ax, threadIdx.x);
    }
    // everything above touches only this CTA's shared memory; from here on global memory written
    // by the kernel before this one is read
    if (kOne && threadIdx.x < sizeof(Req) / 4)
        reinterpret_cast<int*>(sh.reqs)[threadIdx.x] = reinterpret_cast<const int*>(&p.reqs.only)[threadIdx.x];
    grid_dependency_wait();
    const Req* tbl = kOne || p.reqs.n <= kReqCache ? sh.reqs : p.reqs.rows;      // the table is read once per item by every role
    if (!kOne && p.reqs.n <= kReqCache)
#pragma unroll 1
        for (int i = threadIdx.x; i < p.reqs.n * (int)(sizeof(Req) / 4); i += kThreads)
            reinterpret_cast<int*>(sh.reqs)[i] = reinterpret_cast<const int*>(p.reqs.rows)[i];
    if (KIND == kSweep1 && !kSplits && kOne && p.n_clear > 0) {          // no table writer went before
        for (int i = blockIdx.x * kThreads + threadIdx.x; i < p.n_clear; i += gridDim.x * kThreads) p.status[i] = 0;
        write_single_request(p.reqs);
        if (threadIdx.x == kThreads - 1) p.verdicts[blockIdx.x] = LOOKM_OK;  // (a store at the end would hold the launch up)
    }
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&sh.tmem_base), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = sh.tmem_base;
    const int n_cta = gridDim.x;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer ----------
        if (lane == 0) {
            ptx::prefetch_tensormap(&map_a);
            ptx::prefetch_tensormap(&map_b);
            if (KIND == kSweep2) ptx::prefetch_tensormap(&map_x);
            uint32_t gb = 0;                         // streamed tiles armed so far
            int n = 0;                               // stationary tiles armed so far
            bool stop = false;                       // a wait gave up: arm nothing more
            for (int round = 0; !stop; ++round, ++n) {
                const int item = item_of_round(round, blockIdx.x, n_cta);
                if (item >= p.n_items) { if (round * n_cta >= p.n_items) break; --n; continue; }
                const Item it = decode_item<KIND, kSplits, kOne>(p, tbl, item);
                if (kSplits && it.nt == 0) { --n; continue; }
                const int ab = n % kABuf;
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.a_empty[ab]), ((n / kABuf) & 1) ^ 1, abort_flag)) break;
                const uint32_t abar = ptx::smem_u32(&sh.a_full[ab]);
                ptx::mbar_arrive_expect_tx(abar, kTileBytes);
                const uint32_t adst = ptx::smem_u32(&sh.a[ab][0]);
                const int a_row = it.tok_begin + it.blk * kTile;
                ptx::tma_load_3d(adst, &map_a, 0, it.head, a_row, abar);
                ptx::tma_load_3d(adst + kHalfBytes, &map_a, 64, it.head, a_row, abar);
                for (int t = 0; t < it.nt; ++t, ++gb) {
                    const int s = gb % kStages;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.b_empty[s]), ((gb / kStages) & 1) ^ 1, abort_flag)) {
                        stop = true;
                        break;
                    }
                    const uint32_t bbar = ptx::smem_u32(&sh.b_full[s]);
                    ptx::mbar_arrive_expect_tx(bbar, KIND == kSweep2 ? kTileBytes + kSplitBytes : kTileBytes);
                    const uint32_t bdst = ptx::smem_u32(&sh.b[s][0]);
                    if (KIND == kSweep1) {
                        const int row = it.tok_begin + (it.t0 + t) * kTile;
                        const int h = it.head / p.group;
                        ptx::tma_load_3d(bdst, &map_b, 0, h, row, bbar);
                        ptx::tma_load_3d(bdst + kHalfBytes, &map_b, 64, h, row, bbar);
                    } else {
                        const int row = it.tok_begin + (it.blk + (it.t0 + t) / p.group) * kTile;
                        const int h = it.head * p.group + (it.t0 + t) % p.group;
                        ptx::tma_load_3d(bdst, &map_b, 0, h, row, bbar);
                        ptx::tma_load_3d(bdst + kHalfBytes, &map_b, 64, h, row, bbar);
                        ptx::tma_load_3d(ptx::smem_u32(&sh.bx[s % Shared<KIND>::kXStages][0]), &map_x, 0, h, row, bbar);
                    }
                }
            }
            // Every load issued above is consumed by an MMA before the kernel ends, except after an
            // abort.  Then nothing more was armed once a wait had given up (n and gb count exactly
            // the tiles armed), and the copies of the last ring of streamed tiles and of the last two
            // stationary tiles may still be on their way: wait for them (bounded, the flag is
            // ignored; a TMA load completes whether or not anybody consumes it), so that no copy
            // writes shared memory after the CTA has left.
            if (*abort_flag) {
                int ignore = 0;
                for (uint32_t g = (gb > (uint32_t)kStages ? gb - kStages : 0); g < gb; ++g)
                    ptx::mbar_wait(ptx::smem_u32(&sh.b_full[g % kStages]), (g / kStages) & 1, &ignore,
                                   200000000ull);
                for (int m = (n > kABuf ? n - kABuf : 0); m < n; ++m)
                    ptx::mbar_wait(ptx::smem_u32(&sh.a_full[m % kABuf]), (m / kABuf) & 1, &ignore, 200000000ull);
            }
        }
    } else if (warp == 1 || warp == kEpiWarp0 + kGroups * 4) {
        // ------------------------------------------------------------ MMA issuers -----------
        // One thread spends about as long on the waits, fences, commits and loop bookkeeping of a
        // tile as the tensor core needs for its eight MMAs, and it is blocked while they are
        // queued.  Two threads (in warps of different SM sub-partitions) therefore take the tiles
        // alternately: one prepares its next tile while the other one's MMAs run.
        if (lane == 0) {
            const uint32_t me = (warp == 1) ? 0u : 1u;
            constexpr uint32_t idesc = ptx::umma_idesc_bf16(kTile, kTile);
            uint32_t gb = 0;
            int n = 0;
            bool stop = false;                       // a wait gave up: issue nothing more
            for (int round = 0; !stop; ++round, ++n) {
                const int item = item_of_round(round, blockIdx.x, n_cta);
                if (item >= p.n_items) { if (round * n_cta >= p.n_items) break; --n; continue; }
                const Item it = decode_item<KIND, kSplits, kOne>(p, tbl, item);
                if (kSplits && it.nt == 0) { --n; continue; }
                const int ab = n % kABuf;
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.a_full[ab]), (n / kABuf) & 1, abort_flag)) break;
                const uint32_t a_addr = ptx::smem_u32(&sh.a[ab][0]);
                bool issued = false;
                for (int t = 0; t < it.nt; ++t, ++gb) {
                    if ((gb & (kIssuers - 1)) != me) continue;
                    const int s = gb % kStages;
                    const int buf = gb % kAccum;
                    // no MMA is issued on operands that have not landed or into an accumulator that
                    // is still being read
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.b_full[s]), (gb / kStages) & 1, abort_flag) ||
                        !ptx::mbar_wait(ptx::smem_u32(&sh.t_empty[buf]), ((gb / kAccum) & 1) ^ 1, abort_flag)) {
                        stop = true;
                        break;
                    }
                    ptx::tc_fence_after_sync();
                    const uint32_t b_addr = ptx::smem_u32(&sh.b[s][0]);
                    const uint32_t d_tmem = tmem_base + buf * kTile;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        // 16 bf16 (32 bytes) per MMA along the 128-byte swizzled row; the second
                        // half of head_dim lives in the second TMA box.
                        const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
                        ptx::umma_bf16(d_tmem, ptx::umma_desc_sw128(a_addr + off),
                                       ptx::umma_desc_sw128(b_addr + off), idesc, kk > 0);
                    }
                    if (KIND == kSweep2)                 // accumulator += ones x (-lse / scale)^T
                        ptx::umma_bf16(d_tmem, ptx::umma_desc_sw32(ptx::smem_u32(&sh.ax[0])),
                                       ptx::umma_desc_sw32(ptx::smem_u32(&sh.bx[s % Shared<KIND>::kXStages][0])), idesc, 1u);
                    ptx::umma_commit(ptx::smem_u32(&sh.b_empty[s]));
                    ptx::umma_commit(ptx::smem_u32(&sh.t_full[gb % kFullRing]));
                    issued = true;
                }
                if (stop) break;
                // the stationary tile is free when both issuers are through with the item: an
                // issuer that used it arrives when its MMAs have completed, the other one at once
                if (issued) ptx::umma_commit(ptx::smem_u32(&sh.a_empty[ab]));
                else ptx::mbar_arrive(ptx::smem_u32(&sh.a_empty[ab]));
            }
            // Nothing may release TMEM or leave the kernel while an MMA is still running, also
            // after an abort: wait for all of them (own time limit, the abort flag is ignored).
            int ignore = 0;
            ptx::umma_commit(ptx::smem_u32(&sh.mma_done));
            ptx::mbar_wait(ptx::smem_u32(&sh.mma_done), 0, &ignore, 1000000000ull);
        }
    } else {
        // ------------------------------------------------------------ epilogue --------------
        if (KIND == kSweep2 && kOne && blockIdx.x == gridDim.x - 1)  // (not the CTA with the longest item, and its last group first)
            for (int i = 32 * (kEpiWarp0 + 4 * kGroups) - 1 - threadIdx.x; i < p.n_verdicts; i += kGroups * 128)
                if (p.verdicts[i] != LOOKM_OK) atomicExch(p.status, p.verdicts[i]);
        const int wg = (warp - kEpiWarp0) >> 2;              // group of the epilogue
        const int quarter = warp & 3;                        // TMEM lane quarter this warp may read
        const int row = quarter * 32 + lane;                 // row of the stationary tile
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const float c2 = p.scale_log2;
        uint32_t gb = 0;
        int n = 0;
        for (int round = 0;; ++round, ++n) {
            const int item = item_of_round(round, blockIdx.x, n_cta);
            if (item >= p.n_items) { if (round * n_cta >= p.n_items) break; --n; continue; }
            const Item it = decode_item<KIND, kSplits, kOne>(p, tbl, item);
            if (kSplits && it.nt == 0) { --n; continue; }
            const int pos = it.blk * kTile + row;            // position of this thread's row
            float m_run = -INFINITY, l_run = 0.f;            // sweep 1
            float acc[4] = {0.f, 0.f, 0.f, 0.f}, high = -INFINITY;       // sweep 2

            for (int t = 0; t < it.nt; ++t, ++gb) {
                if ((int)(gb % kGroups) != wg) continue;
                const int buf = (int)(gb % kAccum);
                bool diag = false;                           // tile crosses the causal diagonal
                int col_limit = kTile;                       // sweep 2: valid columns of the tile
                int diag_from = 0;                           // sweep 2: first column this row may use
                if (KIND == kSweep1) {
                    diag = (it.t0 + t == it.blk);
                } else {
                    const int ib = it.blk + (it.t0 + t) / p.group;
                    // columns to mask: below the diagonal in the item's first query block, and past
                    // the end of the request in its last one (rows of the next request or zeros)
                    col_limit = min(kTile, it.L - ib * kTile);
                    diag = (ib == it.blk) || (col_limit < kTile);
                    diag_from = (ib == it.blk) ? row : 0;
                }
                ptx::mbar_wait(ptx::smem_u32(&sh.t_full[gb % kFullRing]), (gb / kFullRing) & 1, abort_flag);
                ptx::tc_fence_after_sync();
                // work on 32 columns of the accumulator, c0 = first column of the chunk
                auto process = [&](const uint32_t (&raw)[32], int c0) {
                    if (KIND == kSweep1) {
                        if (diag) sweep1_diagonal(raw, c0, row, c2, m_run, l_run);
                        else sweep1_columns(raw, c2, m_run, l_run);
                    } else {
                        if (diag) sweep2_diagonal(raw, c0, diag_from, col_limit, c2, acc);
                        else sweep2_columns(raw, c2, acc, high);
                    }
                };
                // the last columns are in registers: hand the accumulator back, so that the next
                // tile's MMAs run while this chunk is still being worked on
                auto release = [&]() {
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.t_empty[buf]));
                };
                const uint32_t tbase = lane_addr + buf * kTile;
#pragma unroll 1
                for (int ch = 0; ch < kTile / 32; ++ch) {
                    uint32_t raw[32];
                    ptx::tmem_ld_32x32(tbase + ch * 32, raw);
                    ptx::tmem_ld_wait();
                    if (ch == kTile / 32 - 1) release();
                    process(raw, ch * 32);
                }
            }

            // ---- combine the four groups and write this item's results -----------------------
            // The group that owns the item's last tile finishes last anyway, so it combines: the
            // others leave their partial results in shared memory, signal, and go on to the next
            // item without waiting for anybody.  Values are always combined in group order.
            const int cslot = n & 1;
            const uint32_t cuse = static_cast<uint32_t>(n) >> 1;         // earlier uses of this buffer
            const int combiner = static_cast<int>((gb - 1u) % kGroups);
            float (*cb)[Shared<KIND>::kPlanes][kTile] = sh.comb[cslot];
            constexpr int kP1 = Shared<KIND>::kPlanes - 1;       // second value of a row (not in sweep 2)
            // The buffer's previous contents (two items ago) have been read.  The combining group waits for
            // this too: the parity of comb_full tells one use from the next only once the use before is
            // over, and a warp may come here ahead of others that have yet to arrive for that one (groups
            // without a tile in short items hold nobody back).
            ptx::mbar_wait(ptx::smem_u32(&sh.comb_free[cslot]), (cuse & 1u) ^ 1u, abort_flag);
            if (wg != combiner) {
                if (KIND == kSweep1) { cb[wg][0][row] = m_run; cb[wg][kP1][row] = l_run; }
                else { cb[wg][0][row] = sweep2_sum((acc[0] + acc[1]) + (acc[2] + acc[3]), high, c2); }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_full[cslot]));
            } else {
                ptx::mbar_wait(ptx::smem_u32(&sh.comb_full[cslot]), cuse & 1u, abort_flag);
                if (pos < it.L && !*abort_flag) {
                    if (KIND == kSweep1) {
                        float mg[kGroups], lg[kGroups];
#pragma unroll
                        for (int g = 0; g < kGroups; ++g) {
                            mg[g] = (g == wg) ? m_run : cb[g][0][row];
                            lg[g] = (g == wg) ? l_run : cb[g][kP1][row];
                        }
                        float m = mg[0];
#pragma unroll
                        for (int g = 1; g < kGroups; ++g) m = fmaxf(m, mg[g]);
                        float l = lg[0] * ptx::ex2((mg[0] - m) * c2);
#pragma unroll
                        for (int g = 1; g < kGroups; ++g) l += lg[g] * ptx::ex2((mg[g] - m) * c2);
                        if (kSplits && it.n_splits > 1)
                            __stcg(p.parts1 + ((long long)it.split * p.n_q_heads + it.head) * p.T + it.tok_begin + pos, make_float2(m, l));
                        else
                            store_lse(p, it.head, it.tok_begin + pos, m, l);
                    } else {
                        const float own = sweep2_sum((acc[0] + acc[1]) + (acc[2] + acc[3]), high, c2);
                        float a = (wg == 0) ? own : cb[0][0][row];
#pragma unroll
                        for (int g = 1; g < kGroups; ++g) a += (g == wg) ? own : cb[g][0][row];
                        if (kSplits && it.n_splits > 1)
                            __stcg(p.parts2 + ((long long)it.split * p.n_kv_heads + it.head) * p.T + it.tok_begin + pos, a);
                        else
                            p.scores[(long long)it.head * p.T + it.tok_begin + pos] = a;
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_free[cslot]));
                if (kSplits && it.n_splits > 1) {
                    const int heads = KIND == kSweep1 ? p.n_q_heads : p.n_kv_heads;
                    __threadfence();
                    __syncwarp();
                    int last = 0;
                    if (lane == 0)
                        last = atomicAdd(p.arrived + ((long long)it.tile * heads + it.head) * 4 + quarter, 1) == it.n_splits - 1;
                    if (__shfl_sync(0xffffffffu, last, 0) && pos < it.L && !*abort_flag) {
                        __threadfence();
                        const long long at = (long long)it.head * p.T + it.tok_begin + pos, step = (long long)heads * p.T;
                        if (KIND == kSweep1) {
                            float2 ml[kMaxSplits];
                            float m = -INFINITY, l = 0.f;
#pragma unroll
                            for (int i = 0; i < kMaxSplits; ++i) {
                                ml[i] = i < it.n_splits ? __ldcg(p.parts1 + at + i * step) : make_float2(-INFINITY, 0.f);
                                m = fmaxf(m, ml[i].x);
                            }
#pragma unroll
                            for (int i = 0; i < kMaxSplits; ++i) l += ml[i].y * ptx::ex2((ml[i].x - m) * c2);
                            store_lse(p, it.head, it.tok_begin + pos, m, l);
                        } else {
                            float a = __ldcg(p.parts2 + at);
                            for (int i = 1; i < it.n_splits; ++i) a += __ldcg(p.parts2 + at + i * step);
                            p.scores[at] = a;
                        }
                    }
                }
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && sh.abort_flag)
        atomicExch(KIND == kSweep1 && !kSplits && kOne && p.n_clear > 0 ? p.verdicts + blockIdx.x : p.status, (int)LOOKM_ERR_DEVICE_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------
// The sweeps of large problems: an item owns kBlocks = 2 or 4 adjacent stationary blocks and every
// streamed tile is multiplied with all of them, so a tile is brought into shared memory once per two or
// four products.  These sweeps run at the board's power limit, where time is energy, and a tenth of that
// goes into moving tiles from L2 (a build without the loads ran 9-11 % faster).  Whole layers in a row, ms,
// one block per item | two | four: 16384 tokens x 40 heads 4.45 | 4.10 | 3.92, 32768 x 32 query heads on 8
// 11.2 | 10.6 | 10.4, 8192 x 32 0.918 | 0.886 | 0.93 (the rule: sweep_blocks in api.cu).
// Two blocks: streamed tile g of the CTA goes to accumulators 2 (g mod 2) + block, and each accumulator
// has one issuing thread (g mod 2) and one epilogue group, which works on one block and on the tiles of
// one parity; the two groups of a block are combined at the item's end like the four of tile_kernel.
// Four blocks: one accumulator and one epilogue group each, nothing to combine.  Across the diagonal a
// tile skips the blocks it lies above (sweep 1) or below (sweep 2).
// A CTA starts with the item of its own index and takes further ones from a counter in global memory,
// one ahead of need; the producer passes them on to the other roles through a ring in shared memory.
// Prompts of different lengths come out uneven from a fixed deal (the fullest CTA had 1.17 times the average
// of three prompts of 1800 to 5000 tokens x 32 heads: scores dealt 597 us, by counter 567; 8192 x 32 901 | 889).
// Which CTA takes an item changes no result: a block's tiles are added in their order, two blocks per
// item in the two parities of the tile's index in the item.
// ------------------------------------------------------------------------------------------------
// Items announced to the roles of a CTA, -1: no more.
struct ItemRing {
    unsigned long long full[kItemRing], empty[kItemRing];
    int items[kItemRing];
};
// The n-th announced item; -1 at the end, and after the wait has given up.  For one thread ...
__device__ __forceinline__ int wait_item(ItemRing& ring, int n, volatile int* abort_flag, uint64_t limit_ns = ptx::kWaitLimitNs) {
    if (!ptx::mbar_wait(ptx::smem_u32(&ring.full[n % kItemRing]), (n / kItemRing) & 1, abort_flag, limit_ns)) return -1;
    return *reinterpret_cast<volatile int*>(&ring.items[n % kItemRing]);
}
// ... and for a warp: lane 0 waits and the others follow its verdict (lanes that gave up one by one
// could leave the rest behind in the next warp-wide instruction).
__device__ __forceinline__ int warp_wait_item(ItemRing& ring, int n, volatile int* abort_flag, uint64_t limit_ns = ptx::kWaitLimitNs) {
    int item = 0;
    if ((threadIdx.x & 31) == 0) item = wait_item(ring, n, abort_flag, limit_ns);
    return __shfl_sync(0xffffffffu, item, 0);
}

template <int KIND, int kBlocks>
struct __align__(1024) MultiShared {
    static constexpr int kRing = kBlocks == 2 ? 4 : 2;   // streamed tiles
    static constexpr int kXStages = (KIND == kSweep2) ? kRing : 1;
    static constexpr int kPlanes = (KIND == kSweep2) ? 1 : 2;
    uint8_t a[kBlocks][kTileBytes];              // stationary blocks
    uint8_t b[kRing][kTileBytes];                // streamed tiles
    uint8_t bx[kXStages][kSplitBytes];           // sweep 2: their 16-column companions
    uint8_t ax[kSplitBytes];                     // sweep 2: constant ones tile that multiplies bx
    float comb[2][2][kPlanes][kTile];            // partial results, [buffer][half]
    Req reqs[kReqCache];
    unsigned long long a_full[kBlocks], a_empty[kBlocks];
    unsigned long long b_full[kRing], b_empty[kRing];
    unsigned long long t_full[kAccum], t_empty[kAccum];
    unsigned long long comb_full[2][2], comb_free[2][2];     // [half][buffer]
    unsigned long long mma_done;
    ItemRing ring;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(MultiShared<kSweep1, 2>) + 1024 <= 232448 && sizeof(MultiShared<kSweep2, 2>) + 1024 <= 232448 &&
              sizeof(MultiShared<kSweep1, 4>) + 1024 <= 232448 && sizeof(MultiShared<kSweep2, 4>) + 1024 <= 232448,
              "shared memory of the multi-block sweeps exceeds 227 KB");
static_assert(kAccum == 4 && kGroups == 4 && kIssuers == 2, "the paired sweeps assume this layout");

struct MultiItem {
    int tok_begin, L, blk, head, nt;
    int n;                                       // blocks of the item that exist
    int tile;                                    // index of the first block over the whole batch
    // is streamed tile t multiplied with block b?
    template <int KIND>
    __device__ __forceinline__ bool active(int b, int t) const {
        return b < n && (KIND == kSweep1 ? t <= blk + b : t >= b);
    }
};

// Column sums of one query head for this warp's 32 keys.  With grouped queries they go to memory, and
// the query head of the group that arrives last adds the group in head order.
__device__ __forceinline__ void store_scores(const TileParams& p, int head, int tile, int quarter, int tok, bool mine, float a) {
    if (p.group == 1) {
        if (mine) p.scores[(long long)head * p.T + tok] = a;
        return;
    }
    const int kvh = head / p.group;
    const long long step = (long long)p.n_kv_heads * p.T;
    float* part = p.parts2 + (long long)kvh * p.T + tok;             // of the group's first head
    if (mine) __stcg(part + (head - kvh * p.group) * step, a);
    __threadfence();
    __syncwarp();
    int last = 0;
    if ((threadIdx.x & 31) == 0)
        last = atomicAdd(p.arrived + ((long long)tile * p.n_kv_heads + kvh) * 4 + quarter, 1) == p.group - 1;
    if (!__shfl_sync(0xffffffffu, last, 0) || !mine) return;
    __threadfence();
    float sum = __ldcg(part);
    for (int g = 1; g < p.group; ++g) sum += __ldcg(part + g * step);
    p.scores[(long long)kvh * p.T + tok] = sum;
}

template <int KIND, int kBlocks>
__device__ __forceinline__ MultiItem decode_multi(const TileParams& p, const Req* tbl, int item) {
    // index of the set of kBlocks blocks among the request's, by length (0: the longest)
    const int heads = p.n_q_heads;
    int r, set;
    if (item < p.tail_begin) {
        int lo = 0, hi = p.reqs.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tbl[mid].item_begin[KIND] <= item) lo = mid; else hi = mid - 1;
        }
        r = lo;
        set = (item - tbl[r].item_begin[KIND]) / heads;
    } else {
        const int v = (item - p.tail_begin) / heads;                          // [set][request]
        r = v % p.reqs.n;
        set = (tbl[r].nblk + kBlocks - 1) / kBlocks - p.tail_sets + v / p.reqs.n;
    }
    const Req& rq = tbl[r];
    MultiItem it;
    it.tok_begin = rq.tok_begin;
    it.L = rq.L;
    // Sets are counted from the request's longest blocks on, so that the one that is not full is the shortest.
    // (From the first block on, sweep 1's longest item had a single block where their number is odd. Scores: 2900
    // tokens x 40 heads 130.4 | 127.6 us, 9100 x 32 851 | 844, 12400 x 32 on 8 1482 | 1473, three ragged prompts 548 | 542.)
    const int rest = rq.nblk - kBlocks * set;                                 // blocks from this set on
    it.n = min(kBlocks, rest);
    it.blk = KIND == kSweep1 ? rest - it.n : kBlocks * set;
    it.head = item % heads;          // (the items of a request, and those of the tail, begin at a multiple of it)
    it.tile = rq.tile_begin + it.blk;
    it.nt = KIND == kSweep1 ? it.blk + it.n : rq.nblk - it.blk;
    return it;
}

template <int KIND, int kBlocks>
__global__ void __launch_bounds__(kThreads, 1)
multi_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_x, const TileParams p) {
    extern __shared__ uint8_t smem_raw[];
    typedef MultiShared<KIND, kBlocks> Sh;
    constexpr int kRing = Sh::kRing;
    Sh& sh = *reinterpret_cast<Sh*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile int* abort_flag = &sh.abort_flag;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kBlocks; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.a_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.a_empty[i]), kBlocks == 2 ? kIssuers : 1);      // issuers that use it
        }
        for (int i = 0; i < 2; ++i) {
            for (int j = 0; j < 2; ++j) {
                ptx::mbar_init(ptx::smem_u32(&sh.comb_full[i][j]), 4);
                ptx::mbar_init(ptx::smem_u32(&sh.comb_free[i][j]), 4);
            }
        }
        for (int i = 0; i < kRing; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.b_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.b_empty[i]), kBlocks == 2 ? 1 : kIssuers);
        }
        for (int i = 0; i < kAccum; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.t_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.t_empty[i]), 4);
        }
        ptx::mbar_init(ptx::smem_u32(&sh.mma_done), kIssuers);
        for (int i = 0; i < kItemRing; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.ring.full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.ring.empty[i]), kIssuers + 16);         // MMA threads, epilogue warps
        }
        sh.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (KIND == kSweep2 && threadIdx.x < kTile) write_ones_row(sh.ax, threadIdx.x);
    if (p.reqs.n == 1 && threadIdx.x < sizeof(Req) / 4)          // a single request came with the launch
        reinterpret_cast<int*>(sh.reqs)[threadIdx.x] = reinterpret_cast<const int*>(&p.reqs.only)[threadIdx.x];
    grid_dependency_wait();
    const Req* tbl = p.reqs.n <= kReqCache ? sh.reqs : p.reqs.rows;      // the table is read once per item by every role
    if (p.reqs.n > 1 && p.reqs.n <= kReqCache)
        for (int i = threadIdx.x; i < p.reqs.n * (int)(sizeof(Req) / 4); i += kThreads)
            reinterpret_cast<int*>(sh.reqs)[i] = reinterpret_cast<const int*>(p.reqs.rows)[i];
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&sh.tmem_base), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = sh.tmem_base;
    auto release_item = [&](int n) { ptx::mbar_arrive(ptx::smem_u32(&sh.ring.empty[n % kItemRing])); };

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer ----------
        if (lane == 0) {
            ptx::prefetch_tensormap(&map_a);
            ptx::prefetch_tensormap(&map_b);
            if (KIND == kSweep2) ptx::prefetch_tensormap(&map_x);
            uint32_t gb = 0;                         // streamed tiles armed so far
            uint32_t na[kBlocks] = {};               // stationary blocks armed so far, per place
            bool stop = false;                       // a wait gave up: arm nothing more
            int item = blockIdx.x;                   // the grid has at most n_items CTAs
            for (int n = 0; !stop; ++n) {
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.ring.empty[n % kItemRing]), ((n / kItemRing) & 1) ^ 1, abort_flag)) break;
                sh.ring.items[n % kItemRing] = item < p.n_items ? item : -1;
                ptx::mbar_arrive(ptx::smem_u32(&sh.ring.full[n % kItemRing]));
                if (item >= p.n_items) break;
                const MultiItem it = decode_multi<KIND, kBlocks>(p, tbl, item);
                item = (int)gridDim.x + atomicAdd(p.next_item, 1);   // wanted after this item's loads
                const int kv_head = it.head / p.group;
                const int a_head = KIND == kSweep1 ? it.head : kv_head, b_head = KIND == kSweep1 ? kv_head : it.head;
#pragma unroll
                for (int half = 0; half < kBlocks; ++half) {
                    if (half >= it.n) break;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.a_empty[half]), (na[half] & 1) ^ 1, abort_flag)) { stop = true; break; }
                    const uint32_t bar = ptx::smem_u32(&sh.a_full[half]), dst = ptx::smem_u32(&sh.a[half][0]);
                    const int row = it.tok_begin + (it.blk + half) * kTile;
                    ptx::mbar_arrive_expect_tx(bar, kTileBytes);
                    ptx::tma_load_3d(dst, &map_a, 0, a_head, row, bar);
                    ptx::tma_load_3d(dst + kHalfBytes, &map_a, 64, a_head, row, bar);
                    ++na[half];
                }
                for (int t = 0; t < it.nt && !stop; ++t, ++gb) {
                    const int s = gb % kRing;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.b_empty[s]), ((gb / kRing) & 1) ^ 1, abort_flag)) { stop = true; break; }
                    const uint32_t bar = ptx::smem_u32(&sh.b_full[s]), dst = ptx::smem_u32(&sh.b[s][0]);
                    ptx::mbar_arrive_expect_tx(bar, KIND == kSweep2 ? kTileBytes + kSplitBytes : kTileBytes);
                    const int row = it.tok_begin + (KIND == kSweep1 ? t : it.blk + t) * kTile;
                    ptx::tma_load_3d(dst, &map_b, 0, b_head, row, bar);
                    ptx::tma_load_3d(dst + kHalfBytes, &map_b, 64, b_head, row, bar);
                    if (KIND == kSweep2)
                        ptx::tma_load_3d(ptx::smem_u32(&sh.bx[s % Sh::kXStages][0]), &map_x, 0, b_head, row, bar);
                }
            }
            // after an abort: wait for the copies that may not have been consumed (see tile_kernel)
            if (*abort_flag) {
                int ignore = 0;
                for (uint32_t g = (gb > (uint32_t)kRing ? gb - kRing : 0); g < gb; ++g)
                    ptx::mbar_wait(ptx::smem_u32(&sh.b_full[g % kRing]), (g / kRing) & 1, &ignore, 200000000ull);
#pragma unroll
                for (int half = 0; half < kBlocks; ++half)
                    if (na[half]) ptx::mbar_wait(ptx::smem_u32(&sh.a_full[half]), (na[half] - 1) & 1, &ignore, 200000000ull);
            }
        }
    } else if (warp == 1 || warp == kEpiWarp0 + 16) {
        // ------------------------------------------------------------ MMA issuers -----------
        if (lane == 0) {
            // of two blocks an issuer takes both for the streamed tiles of its parity, of four it takes
            // two for every tile; either way it owns two accumulators
            const uint32_t me = (warp == 1) ? 0u : 1u;
            const int b0 = kBlocks == 2 ? 0 : 2 * (int)me;
            constexpr uint32_t idesc = ptx::umma_idesc_bf16(kTile, kTile);
            uint32_t gb = 0, na[2] = {0, 0}, used[2] = {0, 0};
            bool stop = false;
            for (int n = 0; !stop; ++n) {
                const int item = wait_item(sh.ring, n, abort_flag);
                if (item < 0) break;
                release_item(n);
                const MultiItem it = decode_multi<KIND, kBlocks>(p, tbl, item);
                bool have[2] = {false, false};       // the item's stationary block has been waited for
                for (int t = 0; t < it.nt && !stop; ++t, ++gb) {
                    if (kBlocks == 2 && (gb & 1u) != me) continue;
                    const int s = gb % kRing;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.b_full[s]), (gb / kRing) & 1, abort_flag)) { stop = true; break; }
                    const uint32_t b_addr = ptx::smem_u32(&sh.b[s][0]);
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        if (!it.template active<KIND>(b0 + half, t)) continue;
                        const int acc = 2 * (int)me + half;
                        if ((!have[half] && !ptx::mbar_wait(ptx::smem_u32(&sh.a_full[b0 + half]), na[half] & 1, abort_flag)) ||
                            !ptx::mbar_wait(ptx::smem_u32(&sh.t_empty[acc]), (used[half] & 1) ^ 1, abort_flag)) {
                            stop = true;
                            break;
                        }
                        have[half] = true;
                        ++used[half];
                        ptx::tc_fence_after_sync();
                        const uint32_t a_addr = ptx::smem_u32(&sh.a[b0 + half][0]), d_tmem = tmem_base + acc * kTile;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {
                            const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
                            ptx::umma_bf16(d_tmem, ptx::umma_desc_sw128(a_addr + off), ptx::umma_desc_sw128(b_addr + off), idesc, kk > 0);
                        }
                        if (KIND == kSweep2)             // accumulator += ones x (-lse / scale)^T
                            ptx::umma_bf16(d_tmem, ptx::umma_desc_sw32(ptx::smem_u32(&sh.ax[0])),
                                           ptx::umma_desc_sw32(ptx::smem_u32(&sh.bx[s % Sh::kXStages][0])), idesc, 1u);
                        ptx::umma_commit(ptx::smem_u32(&sh.t_full[acc]));
                    }
                    if (stop) break;
                    ptx::umma_commit(ptx::smem_u32(&sh.b_empty[s]));
                }
                if (stop) break;
                // A stationary block is free when its issuers are through with the item.  An issuer that
                // had no tile for it waits for its arrival all the same: otherwise its arrivals for two
                // items could complete one phase.
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    if (b0 + half >= it.n || stop) continue;
                    if (have[half]) ptx::umma_commit(ptx::smem_u32(&sh.a_empty[b0 + half]));
                    else if (ptx::mbar_wait(ptx::smem_u32(&sh.a_full[b0 + half]), na[half] & 1, abort_flag))
                        ptx::mbar_arrive(ptx::smem_u32(&sh.a_empty[b0 + half]));
                    else stop = true;
                    ++na[half];
                }
            }
            int ignore = 0;                          // no MMA may be running when TMEM is released
            ptx::umma_commit(ptx::smem_u32(&sh.mma_done));
            ptx::mbar_wait(ptx::smem_u32(&sh.mma_done), 0, &ignore, 1000000000ull);
        }
    } else {
        // ------------------------------------------------------------ epilogue --------------
        const int grp = (warp - kEpiWarp0) >> 2;             // = its accumulator
        const int half = kBlocks == 2 ? grp & 1 : grp;       // its block of the item
        const int parity = grp >> 1;                         // two blocks: of the streamed tiles it works on
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t tacc = tmem_base + grp * kTile + (static_cast<uint32_t>(quarter * 32) << 16);
        const float c2 = p.scale_log2;
        uint32_t gb = 0, used = 0, nh = 0;                   // streamed tiles, own tiles, items with this half
        for (int n = 0;; ++n) {
            const int item = warp_wait_item(sh.ring, n, abort_flag);
            if (item < 0) break;
            if (lane == 0) release_item(n);
            const MultiItem it = decode_multi<KIND, kBlocks>(p, tbl, item);
            const uint32_t gb0 = gb;
            gb += it.nt;
            if (half >= it.n) continue;
            const int blk = it.blk + half;
            const int pos = blk * kTile + row;
            const int t_first = KIND == kSweep2 ? half : 0;        // active tiles [t_first, t_end)
            const int t_end = KIND == kSweep1 ? blk + 1 : it.nt;
            float m_run = -INFINITY, l_run = 0.f;            // sweep 1
            float total = 0.f, high = -INFINITY;             // sweep 2: sums of whole tiles (short chains of
                                                             // additions, whatever the prompt's length)
            // tiles of this group: all of them, or the first one of its parity and every other one
            constexpr int kStep = kBlocks == 2 ? 2 : 1;
            int t = t_first + (kBlocks == 2 ? (int)(((gb0 + t_first) ^ parity) & 1u) : 0);
            for (; t < t_end; t += kStep, ++used) {
                ptx::mbar_wait(ptx::smem_u32(&sh.t_full[grp]), used & 1, abort_flag);
                ptx::tc_fence_after_sync();
                bool diag = KIND == kSweep1 && t == blk;
                int col_limit = kTile, diag_from = 0;
                if (KIND == kSweep2) {
                    // columns to mask: below the diagonal, and past the end of the request
                    const int ib = it.blk + t;
                    col_limit = min(kTile, it.L - ib * kTile);
                    diag = ib == blk || col_limit < kTile;
                    diag_from = ib == blk ? row : 0;
                }
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int ch = 0; ch < kTile / 32; ++ch) {
                    uint32_t raw[32];
                    ptx::tmem_ld_32x32(tacc + ch * 32, raw);
                    ptx::tmem_ld_wait();
                    if (ch == kTile / 32 - 1) {              // everything is in registers
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.t_empty[grp]));
                    }
                    if (KIND == kSweep1) {
                        if (diag) sweep1_diagonal(raw, ch * 32, row, c2, m_run, l_run);
                        else sweep1_columns(raw, c2, m_run, l_run);
                    } else {
                        if (diag) sweep2_diagonal(raw, ch * 32, diag_from, col_limit, c2, acc);
                        else sweep2_columns(raw, c2, acc, high);
                    }
                }
                if (KIND == kSweep2) total += (acc[0] + acc[1]) + (acc[2] + acc[3]);
            }
            if (KIND == kSweep2) total = sweep2_sum(total, high, c2);
            if (kBlocks == 4) {                              // nobody else worked on the block
                const bool mine = pos < it.L && !*abort_flag;
                if (KIND == kSweep2) store_scores(p, it.head, it.tile + half, quarter, it.tok_begin + pos, mine, total);
                else if (mine) store_lse(p, it.head, it.tok_begin + pos, m_run, l_run);
                continue;
            }
            // ---- combine the block's two groups: the one with its last tile finishes last ----
            const int buf = nh & 1;
            const uint32_t use = nh >> 1;
            ++nh;
            float (*cb)[kTile] = sh.comb[buf][half & 1];
            constexpr int kP1 = Sh::kPlanes - 1;
            // (both groups wait until the buffer's use before this one is over: see tile_kernel)
            ptx::mbar_wait(ptx::smem_u32(&sh.comb_free[half & 1][buf]), (use & 1u) ^ 1u, abort_flag);
            if ((int)((gb0 + t_end - 1) & 1u) != parity) {
                if (KIND == kSweep1) { cb[0][row] = m_run; cb[kP1][row] = l_run; }
                else cb[0][row] = total;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_full[half & 1][buf]));
            } else {
                ptx::mbar_wait(ptx::smem_u32(&sh.comb_full[half & 1][buf]), use & 1u, abort_flag);
                const bool mine = pos < it.L && !*abort_flag;
                const float other = KIND == kSweep2 ? cb[0][row] : 0.f;
                if (KIND == kSweep1 && mine) {
                    const float m1 = cb[0][row], l1 = cb[kP1][row];
                    const float m = fmaxf(m_run, m1);
                    // (no contraction: the sum must not depend on which group is which)
                    const float l = __fadd_rn(__fmul_rn(l_run, ptx::ex2((m_run - m) * c2)), __fmul_rn(l1, ptx::ex2((m1 - m) * c2)));
                    store_lse(p, it.head, it.tok_begin + pos, m, l);
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_free[half & 1][buf]));
                if (KIND == kSweep2) store_scores(p, it.head, it.tile + half, quarter, it.tok_begin + pos, mine, total + other);
            }
        }
    }

    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && sh.abort_flag) atomicExch(p.status, (int)LOOKM_ERR_DEVICE_TIMEOUT);
}

// The failure path of the bounded waits, exercised without starving a production kernel: thread 0
// waits with ptx::mbar_wait on an mbarrier that nobody arrives at, warp 0's other threads on the same
// barrier see either the limit or the abort flag, the other warps wait like multi_kernel's epilogue for an
// item that nobody announces and must leave together, and the CTA reports the expiry exactly as
// tile_kernel does (shared abort flag -> status word).
__global__ void __launch_bounds__(128)
wait_probe_kernel(unsigned long long limit_ns, int* status) {
    __shared__ unsigned long long bar;
    __shared__ ItemRing ring;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        ptx::mbar_init(ptx::smem_u32(&bar), 1);
        for (int i = 0; i < kItemRing; ++i) ptx::mbar_init(ptx::smem_u32(&ring.full[i]), 1);
        abort_flag = 0;
        ptx::fence_mbar_init();
    }
    __syncthreads();
    volatile int* flag = &abort_flag;
    bool arrived;
    if (threadIdx.x < 32) arrived = ptx::mbar_wait(ptx::smem_u32(&bar), 0, flag, limit_ns);
    else arrived = __any_sync(0xffffffffu, warp_wait_item(ring, 0, flag, limit_ns) >= 0);
    if (__syncthreads_or(arrived)) return;                   // (nobody arrives: the status word then says that nothing expired)
    if (threadIdx.x == 0) atomicExch(status, (int)LOOKM_ERR_DEVICE_TIMEOUT);
}

}  // namespace

cudaError_t launch_wait_probe(unsigned long long limit_ns, int* status, cudaStream_t stream) {
    wait_probe_kernel<<<1, 128, 0, stream>>>(limit_ns, status);
    return cudaGetLastError();
}

cudaError_t launch_tile_kernel(int kind, const CUtensorMap& map_a, const CUtensorMap& map_b,
                               const CUtensorMap* map_x, const TileParams& p, int num_sms,
                               cudaStream_t stream) {
    if (p.n_items <= 0) return cudaSuccess;
    typedef void (*Kernel)(CUtensorMap, CUtensorMap, CUtensorMap, TileParams);
    static const Kernel kernels[2][2][2] = {{{tile_kernel<kSweep1, false, false>, tile_kernel<kSweep1, false, true>},
                                             {tile_kernel<kSweep1, true, false>, tile_kernel<kSweep1, true, true>}},
                                            {{tile_kernel<kSweep2, false, false>, tile_kernel<kSweep2, false, true>},
                                             {tile_kernel<kSweep2, true, false>, tile_kernel<kSweep2, true, true>}}};
    const size_t smem_of[2] = {sizeof(Shared<kSweep1>) + 1024, sizeof(Shared<kSweep2>) + 1024};
    const int grid = tile_grid(p.n_items, num_sms);
    const CUtensorMap& mx = map_x ? *map_x : map_b;      // only sweep 2 uses it
    static const Kernel multi[2][2] = {{multi_kernel<kSweep1, 2>, multi_kernel<kSweep1, 4>},
                                       {multi_kernel<kSweep2, 2>, multi_kernel<kSweep2, 4>}};
    const size_t multi_smem[2][2] = {{sizeof(MultiShared<kSweep1, 2>) + 1024, sizeof(MultiShared<kSweep1, 4>) + 1024},
                                     {sizeof(MultiShared<kSweep2, 2>) + 1024, sizeof(MultiShared<kSweep2, 4>) + 1024}};
    static unsigned long long configured = 0;
    cudaError_t err = once_per_device(configured, [&]() {
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j)
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(multi[i][j], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)multi_smem[i][j]);
        for (int i = 0; i < 2; ++i)
            for (int j = 0; j < 2; ++j)
                for (int one = 0; one < 2; ++one)
                    if (e == cudaSuccess)
                        e = cudaFuncSetAttribute(kernels[i][j][one], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of[i]);
        return e;
    });
    if (err != cudaSuccess) return err;
    if (p.blocks > 1)
        return launch_chained(multi[kind][p.blocks == 4], dim3(grid), dim3(kThreads), multi_smem[kind][p.blocks == 4],
                              stream, map_a, map_b, mx, p);
    return launch_chained(kernels[kind][p.splits > 1][p.reqs.n == 1], dim3(grid), dim3(kThreads), smem_of[kind], stream, map_a, map_b, mx, p);
}

cudaError_t launch_lse_split(const float* lse, int n_q_heads, long long T, float scale_log2,
                             unsigned short* lse_split, const ReqTable& reqs, int* clear, int n_clear, cudaStream_t stream) {
    const long long n = T * n_q_heads;
    if (n <= 0) return cudaSuccess;
    lse_split_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(lse, n_q_heads, T, scale_log2, lse_split, reqs, clear, n_clear);
    return cudaGetLastError();
}

}  // namespace lookm
