// Cosine matching with fused row argmax (Eq. 9): for every evicted key row its nearest kept key.
//
// Persistent, warp-specialised pipeline over 128 x 128 x 128 bf16 tiles, like the sweeps of
// tile_kernels.cu.  A work item owns a STATIONARY block of 128 evicted key rows (the A operand, rows on the
// 128 TMEM lanes), in the order of the evicted list, and streams the tiles of the head's compacted kept
// keys (the B operand) against it.  Each epilogue thread owns one evicted row and keeps the largest
// dot / |kept key| and its slot.
//   warp 0        streamed tiles by TMA, and 1 / |k| of their 128 kept keys by 4-byte cp.async into a ring
//                 of its own (the list of a head begins at any multiple of four bytes)
//   warps 1, 18   one MMA-issuing thread each, streamed tiles taken alternately
//   warps 2-17    four epilogue groups of four warps; group g owns accumulator g and takes the streamed tiles
//                 whose running index is g (mod 4)
//   warp 19       gathers the evicted rows of the stationary blocks, one item ahead of the MMAs
//
// Bound by the issue slots of the epilogue (some 700 per tile and sub-partition: products with 1 / |k|, their maximum,
// and the look-up of its column in most chunks of 32) and by the tensor core, whose operands both come from shared
// memory: 1090 clocks a tile in a steady stream of 26 tiles an item, tensor pipe half busy.  What it took to get
// there, us per call: the norms as part of the streamed tiles instead of a global load, a store and a 128-thread
// barrier before each accumulator; the gathered rows all at once, positions taken four at a time from shared memory
// (with a shuffle or a load per row a block took 14000 clocks, more than an item of 13 tiles lasts); chunks of 32
// columns.  Whole layers, before | now: 4096 tokens x 32 heads 281.4 | 276.6, 4096 x 8 99.3 | 96.7, 8192 x 32 877 | 869.
// Slower: pairs of CTAs on one product (cta_group::2; 8192 x 32 885), two blocks per item (874), looking at a
// chunk's columns only if its largest product times its largest 1 / |k| can beat the best (887: in a warp of 32
// rows there nearly always is one that it can).
#include <cuda_bf16.h>
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace lookm {
namespace {

constexpr int kAccum = 4;                        // TMEM accumulators (128 fp32 columns each) = epilogue groups
constexpr int kIssuers = 2;
constexpr int kEpiWarp0 = 2, kIssuerWarp1 = kEpiWarp0 + 16, kGatherWarp = kIssuerWarp1 + 1;
constexpr int kMatchThreads = 32 * (kGatherWarp + 1);
constexpr int kHalfBytes = kTile * 64 * 2;       // one TMA box: 128 rows x 64 bf16 (128 B rows)
constexpr int kTileBytes = 2 * kHalfBytes;
constexpr int kReqCache = 16;                    // request-table entries cached in shared memory
constexpr int kRing = 4;                         // streamed tiles
// Ring of the kept keys' inverse norms.  An epilogue warp reads tile g's norms until it is through with the
// tile's last columns, after it has handed the accumulator back.  Tile g + 16 is loaded when the MMAs of
// g + 12 are over, so the same group had handed back tile g + 8, which comes after all its work on g.
constexpr int kSideRing = 16;

struct __align__(1024) MatchShared {
    uint8_t a[2][kTileBytes];                    // stationary block: the next item's is gathered while this item's is in use
    uint8_t b[kRing][kTileBytes];                // streamed tiles
    float side[kSideRing][kTile];                // 1 / |k| of the streamed tiles' kept keys
    float comb[2][kAccum][2][kTile];             // partial results of the groups, double-buffered: cosine and slot
    int positions[kTile];                        // of the rows that the gather warp copies
    Req reqs[kReqCache];
    unsigned long long a_full[2], a_empty[2];
    unsigned long long b_full[kRing], b_empty[kRing], side_full[kSideRing];
    unsigned long long t_full[kAccum], t_empty[kAccum];
    unsigned long long comb_full[2], comb_free[2];
    unsigned long long mma_done;
    uint32_t tmem_base;
    int abort_flag;
};
static_assert(sizeof(MatchShared) + 1024 <= 232448, "shared memory of the matching exceeds 227 KB");

struct Item {
    int tok_begin, L, B, E, blk, head, nt;       // blk: block of 128 evicted rows
    long long kept_row0;                         // first row of this (request, head) in the kept-key matrix
    long long ev0;                               // start of its evicted list
};
__device__ __forceinline__ Item decode_item(const TileParams& p, const Req* tbl, int item) {
    int lo = 0, hi = p.reqs.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tbl[mid].item_begin[kMatch] <= item) lo = mid; else hi = mid - 1;
    }
    const Req& rq = tbl[lo];
    const int u = item - rq.item_begin[kMatch];
    Item it;
    it.tok_begin = rq.tok_begin;
    it.L = rq.L;
    it.B = rq.B;
    it.E = rq.E;
    it.head = u % p.n_kv_heads;
    it.blk = u / p.n_kv_heads;
    it.nt = (rq.B + kTile - 1) / kTile;
    it.kept_row0 = rq.kept_off + (long long)it.head * rq.B;
    it.ev0 = rq.ev_off + (long long)it.head * rq.E;
    return it;
}
// Serpentine deal of the item list (longest prompt first); -1: a round in which this CTA has none
__device__ __forceinline__ int item_of_round(int round, int n_items) {
    const int n = gridDim.x, item = round * n + ((round & 1) ? n - 1 - (int)blockIdx.x : (int)blockIdx.x);
    return item < n_items ? item : -1;
}

// The kept tile that an item starts with: the one in which the positions of its rows would lie, because
// neighbouring tokens (of one image) are often the closest keys: the sooner a row meets its best one, the fewer chunks
// of columns take the look-up below (16384 tokens x 40 heads 496 -> 480 us).  Items of at most a tile per group have
// nothing to gain and don't wait for the position.
__device__ __forceinline__ int first_tile(const TileParams& p, const Item& it) {
    if (it.nt <= kAccum) return 0;
    const int e0 = it.blk * kTile;
    const int kept_before = __ldg(p.evict_idx + it.ev0 + e0) - e0;
    return min(max(kept_before / kTile, 0), it.nt - 1);
}

// Running arg-max over 32 columns, of which `limit` count (c0: slot of the first).  The maximum is taken first;
// only when it reaches the running best is its first column looked up.  The lowest slot wins among equals.
__device__ __forceinline__ float max16(const float* w) {
    const float m0 = ptx::fmax3(w[0], w[1], w[2]), m1 = ptx::fmax3(w[3], w[4], w[5]), m2 = ptx::fmax3(w[6], w[7], w[8]),
                m3 = ptx::fmax3(w[9], w[10], w[11]), m4 = ptx::fmax3(w[12], w[13], w[14]);
    return fmaxf(ptx::fmax3(m0, m1, m2), ptx::fmax3(m3, m4, w[15]));
}
__device__ __forceinline__ void best_of_columns(const uint32_t (&raw)[32], const float* side, int c0, int limit, float& best,
                                                int& best_slot) {
    float v[32];
    const float4* sd = reinterpret_cast<const float4*>(side);
#pragma unroll
    for (int c4 = 0; c4 < 8; ++c4) {
        const float4 r4 = sd[c4];
        v[c4 * 4 + 0] = __uint_as_float(raw[c4 * 4 + 0]) * r4.x;
        v[c4 * 4 + 1] = __uint_as_float(raw[c4 * 4 + 1]) * r4.y;
        v[c4 * 4 + 2] = __uint_as_float(raw[c4 * 4 + 2]) * r4.z;
        v[c4 * 4 + 3] = __uint_as_float(raw[c4 * 4 + 3]) * r4.w;
    }
    if (limit < 32) {                            // last tile of the kept list only
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c >= limit) v[c] = -INFINITY;
    }
    const float lo = max16(v), hi = max16(v + 16), mx = fmaxf(lo, hi);
    if (mx >= best && mx > -INFINITY) {
        const bool low = lo == mx;
        int idx = 15;
#pragma unroll
        for (int c = 14; c >= 0; --c)
            if ((low ? v[c] : v[16 + c]) == mx) idx = c;
        idx += c0 + (low ? 0 : 16);
        best_slot = mx > best ? idx : min(best_slot, idx);
        best = mx;
    }
}

__global__ void __launch_bounds__(kMatchThreads, 1)
match_kernel(const __grid_constant__ CUtensorMap map_b, const TileParams p) {
    extern __shared__ uint8_t smem_raw[];
    MatchShared& sh = *reinterpret_cast<MatchShared*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    volatile int* abort_flag = &sh.abort_flag;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.a_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.a_empty[i]), kIssuers);
            ptx::mbar_init(ptx::smem_u32(&sh.comb_full[i]), (kAccum - 1) * 4);    // warps of the other groups
            ptx::mbar_init(ptx::smem_u32(&sh.comb_free[i]), 4);                   // warps of the combining group
        }
        for (int i = 0; i < kRing; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.b_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.b_empty[i]), 1);
        }
        for (int i = 0; i < kSideRing; ++i) ptx::mbar_init(ptx::smem_u32(&sh.side_full[i]), 32);
        for (int i = 0; i < kAccum; ++i) {
            ptx::mbar_init(ptx::smem_u32(&sh.t_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.t_empty[i]), 4);
        }
        ptx::mbar_init(ptx::smem_u32(&sh.mma_done), kIssuers);
        sh.abort_flag = 0;
        ptx::fence_mbar_init();
    }
    if (p.reqs.n == 1 && threadIdx.x < sizeof(Req) / 4)          // a single request came with the launch
        reinterpret_cast<int*>(sh.reqs)[threadIdx.x] = reinterpret_cast<const int*>(&p.reqs.only)[threadIdx.x];
    grid_dependency_wait();
    const Req* tbl = p.reqs.n <= kReqCache ? sh.reqs : p.reqs.rows;      // the table is read once per item by every role
    if (p.reqs.n > 1 && p.reqs.n <= kReqCache)
        for (int i = threadIdx.x; i < p.reqs.n * (int)(sizeof(Req) / 4); i += kMatchThreads)
            reinterpret_cast<int*>(sh.reqs)[i] = reinterpret_cast<const int*>(p.reqs.rows)[i];
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&sh.tmem_base), 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = sh.tmem_base;
    const int rounds = (p.n_items + gridDim.x - 1) / gridDim.x;

    if (warp == 0) {
        // ------------------------------------------------------------ streamed tiles --------
        if (lane == 0) ptx::prefetch_tensormap(&map_b);
        uint32_t gb = 0;                             // streamed tiles armed so far
        bool stop = false;                           // a wait gave up: arm nothing more
        for (int round = 0; round < rounds && !stop; ++round) {
            const int item = item_of_round(round, p.n_items);
            if (item < 0) continue;
            const Item it = decode_item(p, tbl, item);
            int t = first_tile(p, it);
            for (int i = 0; i < it.nt; ++i, ++gb, t = t + 1 < it.nt ? t + 1 : 0) {
                const int s = gb % kRing;
                int free_now = 1;                    // one lane waits, the warp follows its verdict
                if (lane == 0) free_now = ptx::mbar_wait(ptx::smem_u32(&sh.b_empty[s]), ((gb / kRing) & 1) ^ 1, abort_flag) ? 1 : 0;
                if (!__shfl_sync(0xffffffffu, free_now, 0)) { stop = true; break; }
                if (lane == 0) {
                    const uint32_t bar = ptx::smem_u32(&sh.b_full[s]), dst = ptx::smem_u32(&sh.b[s][0]);
                    const int row = (int)(it.kept_row0 + (long long)t * kTile);
                    ptx::mbar_arrive_expect_tx(bar, kTileBytes);
                    ptx::tma_load_2d(dst, &map_b, 0, row, bar);
                    ptx::tma_load_2d(dst + kHalfBytes, &map_b, 64, row, bar);
                }
                const uint32_t sdst = ptx::smem_u32(&sh.side[gb % kSideRing][lane]);
                const float* src = p.rnorm_kept + it.kept_row0;
#pragma unroll
                for (int j = 0; j < kTile / 32; ++j) {
                    const int slot = t * kTile + j * 32 + lane;
                    ptx::cp_async_4(sdst + j * 128, src + (slot < it.B ? slot : 0), slot < it.B ? 4 : 0);
                }
                ptx::cp_async_arrive(ptx::smem_u32(&sh.side_full[gb % kSideRing]));
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        // After an abort nothing more was armed; the copies of the last ring of tiles may still be on
        // their way: wait for them (bounded, the flag is ignored), so that no copy writes shared memory
        // after the CTA has left.  
        if (*abort_flag && lane == 0) {
            int ignore = 0;
            for (uint32_t g = (gb > (uint32_t)kRing ? gb - kRing : 0); g < gb; ++g)
                ptx::mbar_wait(ptx::smem_u32(&sh.b_full[g % kRing]), (g / kRing) & 1, &ignore, 200000000ull);
        }
        __syncwarp();
    } else if (warp == kGatherWarp) {
        // ------------------------------------------------------------ stationary block -------
        // Rows e0 .. e0 + 127 of the head's evicted list, i.e. the key rows at positions evict_idx[e].  Half a warp
        // copies a row of 256 bytes, 16 bytes per lane, lanes 0-15 rows 0-63 of the block and lanes 16-31 rows
        // 64-127, into the layout a TMA box pair with the 128-byte swizzle would have produced: 64 features
        // (128 bytes) per row and box, chunk c of row r at r * 128 + ((c xor (r mod 8)) * 16).  Rows past the
        // end of the list are zero-filled.  The positions go through shared memory, from which a lane takes those of
        // four rows at a time: a shuffle per row, queued behind the epilogue's loads, took 14000 clocks a block.
        const int l16 = lane & 15, r0 = (lane >> 4) * (kTile / 2);
        const uint32_t lane_dst = (l16 >> 3) * kHalfBytes, c8 = l16 & 7;
        int n = 0;
        for (int round = 0; round < rounds; ++round) {
            const int item = item_of_round(round, p.n_items);
            if (item < 0) continue;
            const Item it = decode_item(p, tbl, item);
            const int ab = n & 1;
            const int n_rows = min(kTile, it.E - it.blk * kTile);
            const int* ev = p.evict_idx + it.ev0 + it.blk * kTile;
            int at[kTile / 32];
#pragma unroll
            for (int j = 0; j < kTile / 32; ++j) at[j] = j * 32 + lane < n_rows ? __ldg(ev + j * 32 + lane) : 0;
#pragma unroll
            for (int j = 0; j < kTile / 32; ++j) {
                if (at[j] < 0 || at[j] >= it.L) {
                    atomicExch(p.status, (int)LOOKM_ERR_DEVICE_BAD_INDEX);
                    at[j] = 0;
                }
                sh.positions[j * 32 + lane] = at[j];
            }
            int free_now = 1;
            if (lane == 0) free_now = ptx::mbar_wait(ptx::smem_u32(&sh.a_empty[ab]), ((n >> 1) & 1) ^ 1, abort_flag) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, free_now, 0)) break;
            __syncwarp();                        // the positions are there for all lanes (a shuffle orders no memory)
            ++n;
            const uint32_t adst = ptx::smem_u32(&sh.a[ab][0]) + lane_dst;
            const char* src0 = reinterpret_cast<const char*>(p.k_rows) +
                               2 * ((long long)it.tok_begin * p.k_stride_tok + (long long)it.head * p.k_stride_head) + l16 * 16;
#pragma unroll 4
            for (int st = 0; st < kTile / 2; st += 4) {
                const int4 pos = *reinterpret_cast<const int4*>(&sh.positions[r0 + st]);
                const int four[4] = {pos.x, pos.y, pos.z, pos.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r0 + st + i;
                    ptx::cp_async_16(adst + r * 128 + ((c8 ^ (r & 7)) << 4), src0 + 2 * four[i] * p.k_stride_tok, r < n_rows ? 16 : 0);
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            ptx::fence_proxy_async_shared();
            __syncwarp();                        // (also: the positions have been read)
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.a_full[ab]));
        }
    } else if (warp == 1 || warp == kIssuerWarp1) {
        // ------------------------------------------------------------ MMA issuers -----------
        if (lane == 0) {
            const uint32_t mine = warp == 1 ? 0u : 1u;
            constexpr uint32_t idesc = ptx::umma_idesc_bf16(kTile, kTile);
            uint32_t gb = 0;
            int n = 0;
            bool stop = false;                       // a wait gave up: issue nothing more
            for (int round = 0; round < rounds && !stop; ++round) {
                const int item = item_of_round(round, p.n_items);
                if (item < 0) continue;
                const Item it = decode_item(p, tbl, item);
                const int ab = n & 1;
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.a_full[ab]), (n >> 1) & 1, abort_flag)) break;
                ++n;
                const uint32_t a_addr = ptx::smem_u32(&sh.a[ab][0]);
                bool issued = false;
                for (int t = 0; t < it.nt; ++t, ++gb) {
                    if ((gb & 1u) != mine) continue;
                    const int s = gb % kRing, acc = gb % kAccum;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.b_full[s]), (gb / kRing) & 1, abort_flag) ||
                        !ptx::mbar_wait(ptx::smem_u32(&sh.t_empty[acc]), ((gb / kAccum) & 1) ^ 1, abort_flag)) {
                        stop = true;
                        break;
                    }
                    ptx::tc_fence_after_sync();
                    const uint32_t b_addr = ptx::smem_u32(&sh.b[s][0]), d_tmem = tmem_base + acc * kTile;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)
                        ptx::umma_bf16(d_tmem, ptx::umma_desc_sw128(a_addr + (kk >> 2) * kHalfBytes + (kk & 3) * 32),
                                       ptx::umma_desc_sw128(b_addr + (kk >> 2) * kHalfBytes + (kk & 3) * 32), idesc, kk > 0);
                    ptx::umma_commit(ptx::smem_u32(&sh.b_empty[s]));
                    ptx::umma_commit(ptx::smem_u32(&sh.t_full[acc]));
                    issued = true;
                }
                if (stop) break;
                // the stationary block is free when both issuers are through with the item
                if (issued) ptx::umma_commit(ptx::smem_u32(&sh.a_empty[ab]));
                else ptx::mbar_arrive(ptx::smem_u32(&sh.a_empty[ab]));
            }
            int ignore = 0;                          // no MMA may be running when TMEM is released
            ptx::umma_commit(ptx::smem_u32(&sh.mma_done));
            ptx::mbar_wait(ptx::smem_u32(&sh.mma_done), 0, &ignore, 1000000000ull);
        }
    } else {
        // ------------------------------------------------------------ epilogue --------------
        const int grp = (warp - kEpiWarp0) >> 2;             // = its accumulator
        const int row = (warp & 3) * 32 + lane;              // (a warp may read the TMEM lanes of its quarter)
        const uint32_t tacc = tmem_base + grp * kTile + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        uint32_t gb = 0, used = 0, n = 0;                    // streamed tiles, own tiles, items
        for (int round = 0; round < rounds; ++round) {
            const int item = item_of_round(round, p.n_items);
            if (item < 0) continue;
            const Item it = decode_item(p, tbl, item);
            const uint32_t gb0 = gb;
            gb += it.nt;
            const int e = it.blk * kTile + row;              // index in the evicted list
            float best = -INFINITY;
            int best_slot = 0x7fffffff;
            // 1 / |k| of this thread's evicted row takes two dependent loads (its position, then the norm).
            // They are requested here and after the group's first tile, not in the combine at the item's end,
            // where the group that combines would sit out both round trips while its next accumulator
            // stays full.
            int row_at = 0;
            float row_rnorm = 0.f;
            bool rnorm_asked = false;
            if (e < it.E) row_at = ptx::ld_nc_s32(p.evict_idx + it.ev0 + e);
            const auto ask_rnorm = [&]() {
                if (e < it.E) {
                    int at = row_at;
                    if (at < 0 || at >= it.L) at = 0;       // reported by the gather warp
                    row_rnorm = ptx::ld_nc_f32(p.rnorm_all + (long long)it.head * p.T + it.tok_begin + at);
                }
                rnorm_asked = true;
            };
            const int t0 = first_tile(p, it);
            for (int i = (int)((grp - gb0) & (kAccum - 1)); i < it.nt; i += kAccum, ++used) {
                const uint32_t g = gb0 + i;
                const int t = t0 + i < it.nt ? t0 + i : t0 + i - it.nt;
                const float* side = sh.side[g % kSideRing];
                ptx::mbar_wait(ptx::smem_u32(&sh.side_full[g % kSideRing]), (g / kSideRing) & 1, abort_flag);
                ptx::mbar_wait(ptx::smem_u32(&sh.t_full[grp]), used & 1, abort_flag);
                ptx::tc_fence_after_sync();
                const int limit = it.B - t * kTile;
#pragma unroll 1
                for (int ch = 0; ch < kTile / 32; ++ch) {
                    uint32_t raw[32];
                    ptx::tmem_ld_32x32(tacc + ch * 32, raw);
                    ptx::tmem_ld_wait();
                    if (ch == kTile / 32 - 1) {              // everything is in registers: hand the accumulator back
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.t_empty[grp]));
                    }
                    best_of_columns(raw, side + ch * 32, t * kTile + ch * 32, limit - ch * 32, best, best_slot);
                }
                if (!rnorm_asked) ask_rnorm();
            }
            // ---- combine the groups: the one with the last tile finishes last ------------------
            // The others leave their partial results in shared memory and go on without waiting for anybody.
            // Every group first waits until the buffer's use two items ago is over: parities alone do not
            // tell a warp that runs ahead of its group which use it is looking at.
            const int buf = n & 1;
            const uint32_t use = n >> 1;
            ++n;
            ptx::mbar_wait(ptx::smem_u32(&sh.comb_free[buf]), (use & 1u) ^ 1u, abort_flag);
            if ((int)((gb - 1u) & (kAccum - 1)) != grp) {
                sh.comb[buf][grp][0][row] = best;
                sh.comb[buf][grp][1][row] = __int_as_float(best_slot);
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_full[buf]));
            } else {
                ptx::mbar_wait(ptx::smem_u32(&sh.comb_full[buf]), use & 1u, abort_flag);
                if (e < it.E && !*abort_flag) {
                    if (!rnorm_asked) ask_rnorm();
#pragma unroll
                    for (int i = 0; i < kAccum; ++i) {
                        if (i == grp) continue;
                        const float b1 = sh.comb[buf][i][0][row];
                        const int s1 = __float_as_int(sh.comb[buf][i][1][row]);
                        if (b1 > best || (b1 == best && s1 < best_slot)) { best = b1; best_slot = s1; }
                    }
                    p.assign[it.ev0 + e] = best_slot;
                    p.sim[it.ev0 + e] = best * row_rnorm;
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.comb_free[buf]));
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

}  // namespace

cudaError_t launch_match(const CUtensorMap& map_kept, const TileParams& p, int num_sms, cudaStream_t stream) {
    if (p.n_items <= 0) return cudaSuccess;
    static unsigned long long configured = 0;
    const size_t smem = sizeof(MatchShared) + 1024;
    cudaError_t err = once_per_device(configured, [&]() {
        return cudaFuncSetAttribute(match_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (err != cudaSuccess) return err;
    const int grid = p.n_items < num_sms ? p.n_items : num_sms;
    return launch_chained(match_kernel, dim3(grid), dim3(kMatchThreads), smem, stream, map_kept, p);
}

}  // namespace lookm
