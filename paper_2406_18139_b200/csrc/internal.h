// Internal declarations shared by the host planner (api.cu) and the kernel files.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/lookm.h"

namespace lookm {

constexpr int kTile = 128;      // tokens per tile on either operand of the tensor-core kernels
constexpr int kHeadDim = 128;   // only supported head_dim
constexpr int kMinUnitEntries = 32; // least number of rows in a work unit of the merge kernel
#ifndef LOOKM_MAX_UNIT_ENTRIES
#define LOOKM_MAX_UNIT_ENTRIES 256
#endif
constexpr int kMaxUnitEntries = LOOKM_MAX_UNIT_ENTRIES;   // most rows in one
// Digits of the assignment inversion's radix sort: the slot index of a request with B kept rows is
// split into the fewest digits of at most max_bits bits, all of the same width (so B <= 2^max_bits
// is sorted in one pass).  16-bit counters allow 11-bit digits, 32-bit counters 10-bit ones.
constexpr int kInvDigitBits16 = 11;
constexpr int kInvDigitBits32 = 10;
constexpr int kInvMaxCluster = 8;
// The counting inversion: sixteen warps a CTA, at most kCountSeg evicted rows a warp and kCountMaxSlots
// kept rows, which take kCountSlotBytes of shared memory each.
constexpr int kCountWarps = 16, kCountSeg = 224, kCountMaxSlots = 8192, kCountSlotBytes = 22;
constexpr int kInvWideCountsAbove = 65535;   // evicted tokens per head beyond which counts need 32 bits
#ifdef __CUDACC__
__host__ __device__
#endif
inline void invert_digits(int B, int max_bits, int& n_pass, int& dbits) {
    int bits = 1;
    while ((1 << bits) < B) ++bits;
    n_pass = (bits + max_bits - 1) / max_bits;
    dbits = (bits + n_pass - 1) / n_pass;
}
constexpr int kMergePartBytes = 2560; // per work unit: two fp32 partial K|V rows and one bf16 K|V row

// One request of the packed batch as the kernels see it (device copy lives in the workspace).
// Requests are stored longest first so that the heaviest work items are issued first.
struct Req {
    int tok_begin;        // first token of the request on the packed token axis
    int L;                // prompt length
    int B;                // kept rows  = min(budget, L)
    int M;                // recent window, clamped to B
    int E;                // evicted rows = L - B
    int mode;             // lookm_merge_mode; LOOKM_MERGE_NONE requests have no match items and no
                          // merge work units
    int nblk;             // ceil(L / kTile)
    int out_begin;        // sum of B over the requests before this one (caller order)
    long long kept_off;   // n_kv_heads * out_begin          (start of this request's kept lists)
    long long ev_off;     // n_kv_heads * sum of E before    (start of this request's evicted lists)
    long long sim_off;    // n_kv_heads * sum of E*B before  (start of its similarity blocks)
    long long rp_off;     // kept_off + n_kv_heads * (caller index): start of its scratch of the sorting
                          // inversion, B + 1 words per head
    int item_begin[3];    // first work item of this request in sweep 1 / sweep 2 / match order
    int slot_begin;       // first (head, slot) row of this request in merge order (table order)
    int unit_entries;     // entries read per merge work unit: chosen per call so that every warp
                          // of the merge kernel gets about one unit
    int unit_begin;       // first merge work unit of this request (table order); n_kv_heads *
                          // ceil(L / unit_entries) units per request, heads varying fastest
    int tile_begin;       // 128-row blocks of the requests before this one (table order)
};

// The requests of a call as its launches get them.  A single request travels with every launch: fetching
// it from the table in the workspace would be the first of the dependent loads that a short prompt's kernels
// consist of.
struct ReqTable {
    const Req* rows;      // in the workspace
    int n;
    Req only;             // n == 1
#ifdef __CUDACC__
    __device__ __forceinline__ Req get(int i) const {
        if (n == 1) return only;
        return rows[i];
    }
#endif
};

enum TileKind { kSweep1 = 0, kSweep2 = 1, kMatch = 2 };

constexpr int kMaxSplits = 4;
struct TileParams {
    ReqTable reqs;
    int n_items;
    int n_q_heads, n_kv_heads, group;
    long long T;                 // total packed tokens
    float scale_log2;            // softmax scale * log2(e)
    float* lse;                  // [n_q_heads, T] natural log (sweep 1 writes)
    unsigned short* lse_split;   // [T, n_q_heads, 16] bf16: -lse / scale as three bf16 terms and 13
                                 // zeros per query row (sweep 1 writes, sweep 2 loads it by TMA)
    float* scores;               // [n_kv_heads, T]
    int blocks;                  // blocks per sweep item: 1, or 2 or 4 (multi_kernel; no splits then)
    int splits;                  // ranges that the streamed tiles of a sweep item are cut into
    float2* parts1;              // [splits][n_q_heads, T]  reference and sum of a range (sweep 1)
    float* parts2;               // [splits][n_kv_heads, T] column sums of a range, or of a query head of the
                                 // group (sweep 2)
    int tail_begin, tail_sets;   // multi_kernel: the last items are the shortest tail_sets sets of all requests
    int* next_item;              // items taken beyond the CTAs' first ones (multi_kernel; zeroed)
    int* arrived;                // [block][heads][4] finished ranges per 32 rows (zeroed)
    const int* evict_idx;        // evicted-list layout  (match: rows of the stationary tiles)
    const void* k_rows;          // K [tokens, heads, 128] bf16 with the strides below (match)
    long long k_stride_tok, k_stride_head;
    const float* rnorm_all;      // [n_kv_heads, T]      (match)
    const float* rnorm_kept;     // kept-list layout     (match)
    int* assign;                 // evicted-list layout  (match)
    float* sim;                  // evicted-list layout  (match)
    int* status;                 // device status word
    int n_clear;                 // words from the status word on that sweep 1 has to clear; if any, it also writes the
                                 // single request to its row
    int* verdicts;               // then: one word per CTA of sweep 1, its status.  It can't go to the status word, which
    int n_verdicts;              // another CTA may yet have to clear; sweep 2 passes on what its n_verdicts words say
};

// CTAs of a sweep
inline int tile_grid(int n_items, int num_sms) { return n_items < num_sms ? n_items : num_sms; }

// ---- launchers (each enqueues on `stream` and returns the CUDA error of the launch) -----------
// map_x: the lse_split tensor (sweep 2 only; NULL otherwise)
cudaError_t launch_tile_kernel(int kind, const CUtensorMap& map_a, const CUtensorMap& map_b,
                               const CUtensorMap* map_x, const TileParams& p, int num_sms,
                               cudaStream_t stream);

// Matching of the evicted rows with the compacted kept keys (match_kernel.cu).
cudaError_t launch_match(const CUtensorMap& map_kept, const TileParams& p, int num_sms, cudaStream_t stream);

// lse_split from a given lse (for callers that supply their own log-sum-exp); clears n_clear words from `clear` on and,
// if there are any, writes the single request to its row
cudaError_t launch_lse_split(const float* lse, int n_q_heads, long long T, float scale_log2,
                             unsigned short* lse_split, const ReqTable& reqs, int* clear, int n_clear, cudaStream_t stream);

// One CTA that waits, with the tile kernels' own bounded wait and the given limit, on an mbarrier
// nobody arrives at; on expiry it writes LOOKM_ERR_DEVICE_TIMEOUT to *status like they do.
cudaError_t launch_wait_probe(unsigned long long limit_ns, int* status, cudaStream_t stream);

cudaError_t launch_select(const float* scores, const uint8_t* mask, const ReqTable& reqs,
                          int n_kv_heads, long long T, int max_L, int* kept_idx, int* evict_idx, int* rank,
                          const void* k_for_norms, long long stride_tok, long long stride_head,
                          float* rnorm_all, int num_sms, cudaStream_t stream);

cudaError_t launch_key_norms(const void* k, long long stride_tok, long long stride_head,
                             int n_kv_heads, long long T, float* rnorm_all, cudaStream_t stream);

cudaError_t launch_gather_kept(const void* k, long long stride_tok, long long stride_head,
                               const ReqTable& reqs, int n_kv_heads, long long T,
                               long long total_kept_rows, const int* kept_idx,
                               const float* rnorm_all, void* kept_keys, float* rnorm_kept,
                               int* status, cudaStream_t stream);

cudaError_t launch_argmax_rows(const float* sim_matrix, const ReqTable& reqs, int n_kv_heads,
                               int max_evicted, int* assign, float* sim, cudaStream_t stream);

// Copies up to kReqChunk table entries, passed by value as a kernel argument, into the workspace;
// this keeps the host free of any synchronising copy.
constexpr int kReqChunk = 40;
struct ReqChunk { Req r[kReqChunk]; };
// The launch also zeroes n_clear words from `clear` on (the status word and the counters).
cudaError_t launch_write_table(const ReqChunk& chunk, int count, Req* dst, int* clear, size_t n_clear, cudaStream_t stream);

cudaError_t launch_invert_assignment(const int* assign, const int* kept_idx, const int* evict_idx,
                                     const float* sim, const ReqTable& reqs, int n_kv_heads, int ctas,
                                     long long T, bool wide_counts, int digit_bits, int* row_begin,
                                     int2* entries, int4* unit_first, int* slot_cnt,
                                     unsigned* sort_a, unsigned* sort_b, int* status,
                                     cudaStream_t stream);

cudaError_t launch_invert_counting(const int* assign, const int* kept_idx, const int* evict_idx, const float* sim, const ReqTable& reqs,
                                   int n_kv_heads, int ctas, int max_slots, long long T, int2* entries,
                                   int4* unit_first, int* slot_cnt, int* status, cudaStream_t stream);

// Inversion and merge in one launch; every request has at most kMergeShortMax tokens.
constexpr int kMergeShortMax = 4096;
cudaError_t launch_merge_short(const void* k, const void* v, long long stride_tok, long long stride_head, const int* assign,
                               const int* kept_idx, const int* evict_idx, const float* sim, const ReqTable& reqs,
                               int n_kv_heads, int max_L, int max_E, int max_B, int varlen_output, long long out_stride_head,
                               void* out_k, void* out_v, int* status, int num_sms, cudaStream_t stream);

int merge_warps_per_sm();

cudaError_t launch_merge(const void* k, const void* v, long long stride_tok, long long stride_head,
                         const ReqTable& reqs, int n_kv_heads, long long T,
                         long long total_units, const int2* entries,
                         const int4* unit_first, int* slot_cnt, float* parts,
                         int varlen_output, long long out_stride_head, void* out_k, void* out_v,
                         int num_sms, cudaStream_t stream);

// Kept K and V rows of the requests whose mode is LOOKM_MERGE_NONE copied to the output cache
// (eviction alone, Eq. 6-7); requests with another mode are left to the merge kernel.
cudaError_t launch_compact_kept(const void* k, const void* v, long long stride_tok,
                                long long stride_head, const ReqTable& reqs, int n_kv_heads,
                                long long total_kept_rows, const int* kept_idx, int varlen_output,
                                long long out_stride_head, void* out_k, void* out_v, int* status,
                                cudaStream_t stream);

// ---- generation step over a cache (decode_kernel.cu) --------------------------------------------
// One request of a decode call as the kernel sees it; a launch carries up to kDecodeChunk of them
// by value (no table in device memory, no copy that would synchronise the host).
struct DecodeReq {
    long long begin;      // first cache row of the request
    int len;              // cached rows before the step
    int index;            // position of the request in the caller's q / k_new / v_new / out arrays
    int n_splits;         // CTAs per (KV head, pass)
    int cta_begin;        // first CTA of the request in this launch
    union {
        long long part_begin;   // first partial-result record of the request in the workspace
        long long step_begin;   // shares: steps of the launch before the request's
    };
};
// What a launch gets by value: one request takes 48 bytes, any number up to kDecodeChunk 3088, which costs
// 0.45 us more to launch (409 rows x 32 heads, calls in a row from Python: 6.1 | 5.65 us); up to sixteen, a batch whose
// step may still be as short as its launch, take 528.
constexpr int kDecodeFew = 16;
constexpr int kDecodeChunk = 96;
template <int kRequests>
struct DecodeBatchOf {
    int n_req;
    int share;            // > 0: the CTAs take equal shares of all units' rows, of so many steps each ...
    int longer;           // ... and the first `longer` CTAs one more
    int pad;
    DecodeReq r[kRequests];
};
typedef DecodeBatchOf<kDecodeChunk> DecodeBatch;
static_assert(sizeof(DecodeBatchOf<1>) == 48 && sizeof(DecodeBatchOf<kDecodeFew>) == 528 && sizeof(DecodeBatch) == 3088, "see above");
constexpr int kDecodeShareRows = 64;         // rows of a step
constexpr int kDecodeShareCtasPerSm = 2;

#ifndef LOOKM_DEC_THREADS
#define LOOKM_DEC_THREADS 256
#endif
constexpr int kDecodeThreads = LOOKM_DEC_THREADS;             // threads per CTA of the decode kernel
constexpr int kDecodeMaxCtasPerSm = 2048 / kDecodeThreads;    // more than the kernels' rings let an SM hold
constexpr int kDecodeMaxCluster = 8;     // splits of a (KV head, pass) that one thread-block cluster adds up
int decode_ctas_per_sm(int gt, bool mma);    // resident CTAs per SM of the kernel (0: unknown)

// gt: query heads handled per pass over the rows (divides the group size): 1 or 2, up to 8 on the tensor cores (mma)
// cluster > 1: every request has that many splits, which add up inside the launch
cudaError_t launch_decode(const DecodeBatch& batch, int total_ctas, int gt, bool mma, int cluster, const void* q,
                          const void* k_new, const void* v_new, void* cache_k, void* cache_v,
                          long long stride_row, long long stride_head, int n_q_heads, int n_kv_heads,
                          int rows_per_split, float scale_log2, float* parts, float* out,
                          cudaStream_t stream);
// adds the splits of every request of the batch that has more than one (chained behind launch_decode)
cudaError_t launch_decode_combine(const DecodeBatch& batch, int gt, int n_q_heads, int n_kv_heads,
                                  float scale_log2, const float* parts, float* out, cudaStream_t stream);

// Function attributes (the dynamic shared-memory limit) are set once per device, not per launch:
// `mask` holds one bit per device ordinal on which `configure` has succeeded.  Two threads may both
// run `configure` the first time, which is harmless.
#ifdef __CUDACC__
template <class F>
inline cudaError_t once_per_device(unsigned long long& mask, F configure) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const unsigned long long bit = 1ull << (dev & 63);
    if (__atomic_load_n(&mask, __ATOMIC_ACQUIRE) & bit) return cudaSuccess;
    err = configure();
    if (err == cudaSuccess) __atomic_fetch_or(&mask, bit, __ATOMIC_RELEASE);
    return err;
}
#endif

// Launch with programmatic stream serialisation: the grid may be set up while the kernel before it
// in the stream drains.  Every kernel launched this way starts with grid_dependency_wait(), which
// returns once that kernel has completed and its writes are visible (a no-op for plain launches).
#ifdef __CUDACC__
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained_clusters(void (*kernel)(KArgs...), dim3 grid, dim3 block, unsigned cluster, size_t smem,
                                           cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t stream, Args... args) {
    return launch_chained_clusters(kernel, grid, block, 1u, smem, stream, args...);
}
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif

}  // namespace lookm
