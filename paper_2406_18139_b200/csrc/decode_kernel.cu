// The step after the compression path: one token-generation step of one layer over a (compressed)
// KV cache (Section 3.1, Eq. 2-3).  The new token's K and V rows are appended to the cache and
// every query head attends over its KV head's rows, the new one included:
//     out_g = softmax(q_g K^T * scale) V.
//
// The step is bound by HBM bandwidth: every cached K and V row (256 bytes each) is read exactly
// once per step, whatever the number of query heads in the group, and nothing else of any size
// moves.  The rows of a (request, KV head) are cut into splits of `rows_per_split` rows (chosen
// per call so that the grid is one wave of resident CTAs); a CTA of 8 warps takes one split: half a
// warp owns a row (16 bytes per lane).  Rows travel global -> shared memory with 16-byte cp.async
// copies into a ring private to each warp (a step = four K and four V rows per half-warp; the
// steps ahead are in flight while one is worked on, and every lane reads back exactly the bytes it
// copied, so cp.async.wait_group is all the synchronisation there is).  The dot products are
// reduced with four shuffles, and each half-warp keeps its own running softmax statistics
// (reference maximum, sum, weighted V sum) for every query head of the group in registers.  Half-warps and warps are combined through shared memory in a fixed order; with more
// than one split the CTA leaves its partial result in the workspace and a second kernel, chained
// behind the first, adds the splits in split order.  No CTA waits for another and the order of
// additions never depends on timing, so results are reproducible bit for bit.
//
// Batches whose caches differ much in length, or have few rows, and head counts that leave SMs without a split
// go to decode_shared_kernel below, whose CTAs take equal shares of the rows of all units.
//
// Several query heads that share a KV head can go to decode_mma_kernel below, which has the same structure;
// the planner compares (decode_way in api.cu).
#include <cuda_bf16.h>
#include <float.h>
#include <math.h>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"

namespace lookm {
namespace {

constexpr int kDecThreads = kDecodeThreads;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecHalfWarps = 2 * kDecWarps;         // rows a CTA has in hand at once
#ifndef LOOKM_DEC_FLIGHT
#define LOOKM_DEC_FLIGHT 4
#endif
#ifndef LOOKM_DEC_RING
#define LOOKM_DEC_RING 4
#endif
constexpr int kDecFlight = LOOKM_DEC_FLIGHT;         // rows per half-warp and step
constexpr int kDecRing = LOOKM_DEC_RING;             // steps in the ring of a warp (all but one in flight)
constexpr int kDecRowBytes = kHeadDim * 2;
constexpr int kDecStepBytes = 2 * kDecFlight * 2 * kDecRowBytes;   // per warp: [half][row][K|V][256 B]
constexpr int kDecRingBytes = kDecWarps * kDecRing * kDecStepBytes;

__device__ __forceinline__ void unpack_bf16x8(const uint4& u, float (&x)[8]) {
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i] = __uint_as_float(w[i] << 16);
        x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
}

__device__ __forceinline__ float dec_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Clusters: for short caches all splits of a (request, KV head, pass) are the CTAs of one thread-block
// cluster, which add their results through distributed shared memory, so that no second kernel and no
// partial results in memory are needed.

// What a CTA leaves for the cluster: per query head of the pass reference, sum and weighted V sum.
template <int GP>
struct ClusterShared {
    float m[GP], l[GP];
    float o[GP][kHeadDim];
};
// Adds the n splits of the cluster in split order; every CTA writes its share of the features of gt
// heads.
template <int GP>
__device__ __forceinline__ void cluster_combine(const ClusterShared<GP>& cs, int n, int gt, float scale_log2, float* out) {
    ptx::cluster_sync();
    const int share = kHeadDim / n;
    for (int i = threadIdx.x; i < gt * share; i += blockDim.x) {
        const int g = i / share, t = (int)ptx::cluster_rank() * share + i % share;
        float m[kDecodeMaxCluster], l[kDecodeMaxCluster], o[kDecodeMaxCluster];
        float mx = -INFINITY;
#pragma unroll
        for (int c = 0; c < kDecodeMaxCluster; ++c) {
            m[c] = -INFINITY;
            l[c] = o[c] = 0.f;
            if (c < n) {
                m[c] = ptx::ld_cluster(&cs.m[g], c);
                l[c] = ptx::ld_cluster(&cs.l[g], c);
                o[c] = ptx::ld_cluster(&cs.o[g][t], c);
            }
        }
#pragma unroll
        for (int c = 0; c < kDecodeMaxCluster; ++c) mx = fmaxf(mx, m[c]);
        float lsum = 0.f, osum = 0.f;
#pragma unroll
        for (int c = 0; c < kDecodeMaxCluster; ++c) {
            const float a = m[c] == -INFINITY ? 0.f : dec_ex2((m[c] - mx) * scale_log2);       // a split may be empty
            lsum = fmaf(l[c], a, lsum);
            osum = fmaf(o[c], a, osum);
        }
        out[(long long)g * kHeadDim + t] = osum / lsum;
    }
    ptx::cluster_sync();                                  // nobody leaves while its shared memory is read
}

template <int GT>
struct DecShared {
    float m[kDecWarps][GT];                          // [warp][query head of the pass]
    float l[kDecWarps][GT];
    float o[kDecWarps][GT][kHeadDim];
};

// Asks for the first rows of a CTA's split while the kernel before this one drains: rows already in the cache
// may not be read before that kernel is over, but they may be brought into L2.  It helps behind a kernel that lets its
// dependents start early (this library's do) and is within the scatter behind one that does not.  Caches in rotation, us per
// step without | with, step after step and with a framework's elementwise kernel before each: 8192 rows x 32 heads 23.7 | 23.3,
// 27.4 | 27.4; 32768 x 32 on 8 27.6 | 27.1, 30.9 | 30.9; 20000 x 8 18.2 | 17.6, 21.6 | 21.2; 1638 x 32 8.2 | 7.8, 11.7 | 12.0.
// Of splits of 384 rows and more, 96 rows: asking for 256 of them gains nothing, for 512 costs 1 us.
constexpr int kPrefetchRows = 96, kPrefetchFrom = 384;
__device__ __forceinline__ void prefetch_rows(const __nv_bfloat16* cache_k, const __nv_bfloat16* cache_v, long long first,
                                              long long stride_row, int rows) {
    if (rows < kPrefetchFrom) return;
    for (int i = threadIdx.x; i < kPrefetchRows * 2; i += blockDim.x) {
        const long long at = first + (long long)(i >> 1) * stride_row + (i & 1) * 64;
        ptx::prefetch_l2(cache_k + at);
        ptx::prefetch_l2(cache_v + at);
    }
}

// A half-warp's query features and running softmax statistics (reference, sum, weighted V sum); a lane has 8
// features.
template <int GT>
struct DecState {
    float qv[GT][8], m[GT], l[GT], o[GT][8];
    __device__ __forceinline__ void reset() {
#pragma unroll
        for (int g = 0; g < GT; ++g) {
            m[g] = -INFINITY;
            l[g] = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) o[g][i] = 0.f;
        }
    }
    // q: this lane's features of the pass's first head
    __device__ __forceinline__ void load_query(const __nv_bfloat16* q) {
#pragma unroll
        for (int g = 0; g < GT; ++g) unpack_bf16x8(*reinterpret_cast<const uint4*>(q + g * kHeadDim), qv[g]);
    }
    // One step's rows, K and V alternating from shared address src on, the f-th of them at position row + f *
    // kDecHalfWarps: online softmax against the running maximum of this half-warp.  Rows from row1 on don't count.
    __device__ __forceinline__ void take(uint32_t src, int row, int row1, float scale_log2) {
        uint4 ku[kDecFlight], vu[kDecFlight];
#pragma unroll
        for (int f = 0; f < kDecFlight; ++f) {
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(ku[f].x), "=r"(ku[f].y), "=r"(ku[f].z), "=r"(ku[f].w)
                         : "r"(src + (2 * f) * kDecRowBytes));
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(vu[f].x), "=r"(vu[f].y), "=r"(vu[f].z), "=r"(vu[f].w)
                         : "r"(src + (2 * f + 1) * kDecRowBytes));
        }
        float s[kDecFlight][GT];
#pragma unroll
        for (int f = 0; f < kDecFlight; ++f) {
            const bool valid = row + f * kDecHalfWarps < row1;
            float kx[8];
            unpack_bf16x8(ku[f], kx);
#pragma unroll
            for (int g = 0; g < GT; ++g) {
                float d = 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) d = fmaf(qv[g][i], kx[i], d);
#pragma unroll
                for (int ofs = 8; ofs > 0; ofs >>= 1) d += __shfl_xor_sync(0xffffffffu, d, ofs, 16);
                s[f][g] = valid ? d : -INFINITY;
            }
        }
#pragma unroll
        for (int g = 0; g < GT; ++g) {
            float mx = m[g];
#pragma unroll
            for (int f = 0; f < kDecFlight; ++f) mx = fmaxf(mx, s[f][g]);
            if (mx == -INFINITY) continue;                       // no valid row for this half-warp yet
            const float alpha = dec_ex2((m[g] - mx) * scale_log2);   // 0 when m was -inf
            float p[kDecFlight], ps = 0.f;
#pragma unroll
            for (int f = 0; f < kDecFlight; ++f) {
                p[f] = dec_ex2((s[f][g] - mx) * scale_log2);     // 0 for an invalid row
                ps += p[f];
            }
            l[g] = l[g] * alpha + ps;
            m[g] = mx;
#pragma unroll
            for (int i = 0; i < 8; ++i) o[g][i] *= alpha;
#pragma unroll
            for (int f = 0; f < kDecFlight; ++f) {
                float vx[8];
                unpack_bf16x8(vu[f], vx);
#pragma unroll
                for (int i = 0; i < 8; ++i) o[g][i] = fmaf(p[f], vx[i], o[g][i]);
            }
        }
    }
    // Combines the two half-warps of a warp and leaves the result for the CTA.
    __device__ __forceinline__ void leave(DecShared<GT>& sh, int warp, int lane, float scale_log2) {
#pragma unroll
        for (int g = 0; g < GT; ++g) {
            const float m_o = __shfl_xor_sync(0xffffffffu, m[g], 16);
            const float l_o = __shfl_xor_sync(0xffffffffu, l[g], 16);
            const float mx = fmaxf(m[g], m_o);
            // lower half-warp first, whichever half this lane is in
            const bool low = lane < 16;
            const float a_me = (mx == -INFINITY) ? 0.f : dec_ex2((m[g] - mx) * scale_log2);
            const float a_ot = (mx == -INFINITY) ? 0.f : dec_ex2((m_o - mx) * scale_log2);
            const float l_lo = low ? l[g] * a_me : l_o * a_ot, l_hi = low ? l_o * a_ot : l[g] * a_me;
            l[g] = l_lo + l_hi;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float o_o = __shfl_xor_sync(0xffffffffu, o[g][i], 16);
                const float o_lo = low ? o[g][i] * a_me : o_o * a_ot, o_hi = low ? o_o * a_ot : o[g][i] * a_me;
                o[g][i] = o_lo + o_hi;
            }
            m[g] = mx;
            if (lane == 0) { sh.m[warp][g] = m[g]; sh.l[warp][g] = l[g]; }
            if (low) {
#pragma unroll
                for (int i = 0; i < 8; ++i) sh.o[warp][g][(lane & 15) * 8 + i] = o[g][i];
            }
        }
    }
};
// The warps' results of query head g in warp order: reference, sum and weighted V sum of feature t.
template <int GT>
__device__ __forceinline__ void add_warps(const DecShared<GT>& sh, int g, int t, float scale_log2, float& mx, float& lsum, float& osum) {
    mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) mx = fmaxf(mx, sh.m[w][g]);
    lsum = osum = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
        const float a = mx == -INFINITY ? 0.f : dec_ex2((sh.m[w][g] - mx) * scale_log2);   // 0 for an idle warp
        lsum = fmaf(sh.l[w][g], a, lsum);
        osum = fmaf(sh.o[w][g][t], a, osum);
    }
}

// GT = 1 or 2 query heads of the group are handled per pass over the rows.
template <class Batch, int GT, bool kClustered>
__global__ void __launch_bounds__(kDecThreads)
decode_kernel(const __grid_constant__ Batch batch, const __nv_bfloat16* __restrict__ q,
              const __nv_bfloat16* __restrict__ k_new, const __nv_bfloat16* __restrict__ v_new,
              __nv_bfloat16* __restrict__ cache_k, __nv_bfloat16* __restrict__ cache_v,
              long long stride_row, long long stride_head, int n_q_heads, int n_kv_heads, int group,
              int rows_per_split, float scale_log2, float* __restrict__ parts, float* __restrict__ out) {
    __shared__ DecShared<GT> sh;
    __shared__ ClusterShared<GT> cs;
    extern __shared__ __align__(128) uint8_t dec_ring[];         // [warp][ring step][half][row][K|V][256 B]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hw = threadIdx.x >> 4, l16 = lane & 15;

    // which (request, KV head, pass, split) this CTA owns: requests are found by their first CTA
    int r = 0;
    {
        int lo = 0, hi = batch.n_req - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (batch.r[mid].cta_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        r = lo;
    }
    const DecodeReq rq = batch.r[r];
    const int n_pass = group / GT;
    const int local = (int)blockIdx.x - rq.cta_begin;            // [head][pass][split]
    const int split = local % rq.n_splits;
    const int pass = (local / rq.n_splits) % n_pass;
    const int h = local / (rq.n_splits * n_pass);
    const int n_rows = rq.len + 1;                               // cached rows + the new one
    const int row0 = split * rows_per_split, row1 = min(n_rows, row0 + rows_per_split);
    const int qh0 = h * group + pass * GT;                       // first query head of this pass

    prefetch_rows(cache_k, cache_v, (rq.begin + row0) * stride_row + h * stride_head, stride_row, min(row1, rq.len) - row0);
    grid_dependency_wait();

    DecState<GT> state;
    state.load_query(q + ((long long)rq.index * n_q_heads + qh0) * kHeadDim + l16 * 8);
    state.reset();
    const long long head_off = (long long)h * stride_head + l16 * 8;
    const __nv_bfloat16* ck = cache_k + rq.begin * stride_row + head_off;
    const __nv_bfloat16* cv = cache_v + rq.begin * stride_row + head_off;
    const __nv_bfloat16* nk = k_new + ((long long)rq.index * n_kv_heads + h) * kHeadDim + l16 * 8;
    const __nv_bfloat16* nv = v_new + ((long long)rq.index * n_kv_heads + h) * kHeadDim + l16 * 8;

    // The appended row (Eq. 2) is read from k_new / v_new by whoever owns it; the CTA that owns it
    // on the group's first pass also writes it into the cache (nobody reads cache row `len` in this
    // step, so the write races with nothing).
    if (pass == 0 && rq.len >= row0 && rq.len < row1 && warp == 0) {
        const __nv_bfloat16* src = lane < 16 ? nk : nv;
        __nv_bfloat16* dst = (lane < 16 ? cache_k : cache_v) + rq.begin * stride_row + head_off +
                             (long long)rq.len * stride_row;
        *reinterpret_cast<uint4*>(dst) = __ldg(reinterpret_cast<const uint4*>(src));
    }

    // Copies of one step: K and V of kDecFlight rows per half-warp, 16 bytes per lane and row,
    // straight into this warp's ring.  Rows past the split are zero-filled (a copy of 0 source
    // bytes), so that they contribute exact zeros.  One commit group per step, also past the end.
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(dec_ring) + warp * (kDecRing * kDecStepBytes) +
                           ((lane >> 4) * kDecFlight * 2) * kDecRowBytes + l16 * 16;
    auto issue = [&](int step) {
        const int base = row0 + step * (kDecHalfWarps * kDecFlight);
        const uint32_t dst = ring0 + (uint32_t)(step % kDecRing) * kDecStepBytes;
        if (base < row1) {
#pragma unroll
            for (int f = 0; f < kDecFlight; ++f) {
                const int row = base + f * kDecHalfWarps + hw;
                const bool is_new = (row == rq.len);
                const bool valid = row < row1;
                const __nv_bfloat16* kp = (is_new || !valid) ? nk : ck + (long long)row * stride_row;
                const __nv_bfloat16* vp = (is_new || !valid) ? nv : cv + (long long)row * stride_row;
                const int nbytes = valid ? 16 : 0;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                             ::"r"(dst + (2 * f) * kDecRowBytes), "l"(kp), "r"(nbytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                             ::"r"(dst + (2 * f + 1) * kDecRowBytes), "l"(vp), "r"(nbytes) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the step count does not depend on the half-warp, so both halves of a warp reach the shuffles
    const int n_steps = (row1 - row0 + kDecHalfWarps * kDecFlight - 1) / (kDecHalfWarps * kDecFlight);
#pragma unroll
    for (int st = 0; st < kDecRing - 1; ++st) issue(st);
    for (int st = 0; st < n_steps; ++st) {
        // the buffer refilled here was read into registers one iteration ago
        issue(st + kDecRing - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kDecRing - 1) : "memory");
        state.take(ring0 + (uint32_t)(st % kDecRing) * kDecStepBytes, row0 + st * (kDecHalfWarps * kDecFlight) + hw, row1, scale_log2);
    }

    // ---- combine: the two half-warps of a warp in registers, then the warps in warp order -------
    state.leave(sh, warp, lane, scale_log2);
    __syncthreads();
    // thread t < 128 owns feature t of every query head of the pass
    const int n_splits = rq.n_splits;
    const long long part_stride = kHeadDim + 2;                  // m, l, o[128]
    float* my_parts = parts + ((long long)rq.part_begin + ((long long)(h * n_pass + pass) * n_splits + split) * GT) * part_stride;
    if (threadIdx.x < kHeadDim) {
        const int t = threadIdx.x;
#pragma unroll
        for (int g = 0; g < GT; ++g) {
            float mx, lsum, osum;
            add_warps(sh, g, t, scale_log2, mx, lsum, osum);
            if (kClustered) {
                if (t == 0) { cs.m[g] = mx; cs.l[g] = lsum; }
                cs.o[g][t] = osum;
            } else if (n_splits == 1) {
                out[((long long)rq.index * n_q_heads + qh0 + g) * kHeadDim + t] = osum / lsum;
            } else {
                float* rec = my_parts + g * part_stride;
                if (t == 0) { rec[0] = mx; rec[1] = lsum; }
                rec[2 + t] = osum;
            }
        }
    }
    if (kClustered)
        cluster_combine(cs, n_splits, GT, scale_log2, out + ((long long)rq.index * n_q_heads + qh0) * kHeadDim);
}

// ---------------------------------------------------------------------------------------------
// One query head at a time, equal shares.  The rows of all units ((request, query head), a unit's rows in steps of
// 64) form one sequence, and every CTA takes the same number of steps of it, two CTAs to an SM: a CTA may
// end one unit and begin the next, and its copies run ahead into the next unit while it combines.  A unit that
// lies in several CTAs' shares is added up by decode_combine_kernel; a CTA leaves at most two partial results
// (of the unit its share begins in and of the one it ends in).
// us per step, whole splits | shares: four caches of 1000 to 8000 rows x 32 heads 75.7 | 47.5, 64 of 40 rows x 32 38.0 | 18.3,
// one of 32768 x 40 117 | 108, one of 4000 x 76 38.7 | 29.5; but 20000 x 8 18.4 | 20.8, and nine of 61 to 4390 x 32 60.7 | 86.5:
// a share's units cost some 0.9 us each beside their rows (the planner compares: decode_way in api.cu).
// ---------------------------------------------------------------------------------------------
constexpr int kShareRing = 3;                        // steps in the ring of a warp: two CTAs to an SM
constexpr int kShareRingBytes = kDecWarps * kShareRing * kDecStepBytes;
constexpr int kShareRows = kDecHalfWarps * kDecFlight;
static_assert(kShareRows == kDecodeShareRows, "the planner counts these steps");
static_assert(kShareRingBytes * (kDecodeShareCtasPerSm + 1) > (228 << 10) && 2 * kDecodeShareCtasPerSm <= kDecodeMaxCtasPerSm,
              "the workspace has room for two partial results of every CTA");

// A CTA's way through its share.
struct Walk {
    int r, h;                                        // request; query head
    int row, row1;                                   // next row; end of the share's part of the unit
    int left;                                        // the CTA's steps from here on
};
__device__ __forceinline__ int unit_steps(const DecodeReq& rq) { return rq.len / kShareRows + 1; }       // of len + 1 rows
__device__ __forceinline__ long long divide(long long x, int y) { return x >> 31 ? x / y : (int)x / y; }
// First step of CTA c's share, and the CTA that has a given step: every share has batch.share steps, the first
// batch.longer shares one more.
template <class Batch>
__device__ __forceinline__ long long share_begin(const Batch& batch, int c) {
    return (long long)c * batch.share + min(c, batch.longer);
}
template <class Batch>
__device__ __forceinline__ int share_of(const Batch& batch, long long step) {
    const long long in_longer = (long long)batch.longer * (batch.share + 1);
    return step < in_longer ? (int)divide(step, batch.share + 1) : batch.longer + (int)divide(step - in_longer, batch.share);
}
template <class Batch>
__device__ __forceinline__ Walk start_walk(const Batch& batch) {
    const long long s0 = share_begin(batch, blockIdx.x);
    int lo = 0, hi = batch.n_req - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (batch.r[mid].step_begin <= s0) lo = mid; else hi = mid - 1;
    }
    const DecodeReq& rq = batch.r[lo];
    const int n = unit_steps(rq);
    Walk w;
    w.r = lo;
    w.h = (int)divide(s0 - rq.step_begin, n);
    const int st = (int)(s0 - rq.step_begin - (long long)w.h * n);
    w.left = batch.share + ((int)blockIdx.x < batch.longer ? 1 : 0);
    w.row = st * kShareRows;
    w.row1 = w.left >= n - st ? rq.len + 1 : (st + w.left) * kShareRows;
    return w;
}
// On to the next step; true if it belongs to another unit.
template <class Batch>
__device__ __forceinline__ bool next_step(Walk& w, const Batch& batch, int n_q_heads) {
    --w.left;
    w.row += kShareRows;
    if (w.row < w.row1 || w.left == 0) return false;
    if (++w.h == n_q_heads) { w.h = 0; ++w.r; }
    const DecodeReq& rq = batch.r[w.r];
    w.row = 0;
    w.row1 = w.left >= unit_steps(rq) ? rq.len + 1 : w.left * kShareRows;
    return true;
}

template <class Batch>
__global__ void __launch_bounds__(kDecThreads)
decode_shared_kernel(const __grid_constant__ Batch batch, const __nv_bfloat16* __restrict__ q,
                     const __nv_bfloat16* __restrict__ k_new, const __nv_bfloat16* __restrict__ v_new,
                     __nv_bfloat16* __restrict__ cache_k, __nv_bfloat16* __restrict__ cache_v,
                     long long stride_row, long long stride_head, int n_q_heads, int n_kv_heads, int group,
                     float scale_log2, float* __restrict__ parts, float* __restrict__ out) {
    __shared__ DecShared<1> shared_parts[2];         // of the last part of a unit and the one before
    extern __shared__ __align__(128) uint8_t dec_ring[];         // [warp][ring step][half][row][K|V][256 B]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hw = threadIdx.x >> 4, l16 = lane & 15;

    Walk ahead = start_walk(batch);                  // the copies' way
    {
        const DecodeReq& rq = batch.r[ahead.r];
        prefetch_rows(cache_k, cache_v, (rq.begin + ahead.row) * stride_row + (long long)(ahead.h / group) * stride_head, stride_row,
                      min(ahead.row1, rq.len) - ahead.row);
    }
    grid_dependency_wait();

    const __nv_bfloat16 *ck, *cv, *nk, *nv;
    int len;
    const auto enter = [&]() {
        const DecodeReq& rq = batch.r[ahead.r];
        const int kvh = ahead.h / group;
        const long long off = rq.begin * stride_row + (long long)kvh * stride_head + l16 * 8;
        const long long row_new = ((long long)rq.index * n_kv_heads + kvh) * kHeadDim + l16 * 8;
        ck = cache_k + off;
        cv = cache_v + off;
        nk = k_new + row_new;
        nv = v_new + row_new;
        len = rq.len;
    };
    enter();
    // copies of one step, as in decode_kernel
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(dec_ring) + warp * (kShareRing * kDecStepBytes) +
                           ((lane >> 4) * kDecFlight * 2) * kDecRowBytes + l16 * 16;
    const auto issue = [&](int step) {
        const uint32_t dst = ring0 + (uint32_t)(step % kShareRing) * kDecStepBytes;
        if (ahead.left > 0) {
#pragma unroll
            for (int f = 0; f < kDecFlight; ++f) {
                const int row = ahead.row + f * kDecHalfWarps + hw;
                const bool is_new = (row == len);
                const bool valid = row < ahead.row1;
                const __nv_bfloat16* kp = (is_new || !valid) ? nk : ck + (long long)row * stride_row;
                const __nv_bfloat16* vp = (is_new || !valid) ? nv : cv + (long long)row * stride_row;
                ptx::cp_async_16(dst + (2 * f) * kDecRowBytes, kp, valid ? 16 : 0);
                ptx::cp_async_16(dst + (2 * f + 1) * kDecRowBytes, vp, valid ? 16 : 0);
            }
            if (next_step(ahead, batch, n_q_heads)) enter();
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Walk here = ahead;                               // the arithmetic's way
#pragma unroll
    for (int st = 0; st < kShareRing - 1; ++st) issue(st);

    DecState<1> state;
    const auto begin_part = [&]() {
        const DecodeReq& rq = batch.r[here.r];
        state.load_query(q + ((long long)rq.index * n_q_heads + here.h) * kHeadDim + l16 * 8);
        state.reset();
        // whoever owns the appended row for the group's first head also writes it into the cache
        if (here.h % group == 0 && rq.len >= here.row && rq.len < here.row1 && warp == 0) {
            const long long from = ((long long)rq.index * n_kv_heads + here.h / group) * kHeadDim + l16 * 8;
            const long long to = (rq.begin + rq.len) * stride_row + (long long)(here.h / group) * stride_head + l16 * 8;
            *reinterpret_cast<uint4*>((lane < 16 ? cache_k : cache_v) + to) =
                __ldg(reinterpret_cast<const uint4*>((lane < 16 ? k_new : v_new) + from));
        }
    };
    begin_part();
    bool from_start = here.row == 0;                 // the part begins with its unit
    int part = 0;                                    // parts of units so far
    for (int st = 0; here.left > 0; ++st) {
        issue(st + kShareRing - 1);                  // the buffer refilled here was read into registers one iteration ago
        asm volatile("cp.async.wait_group %0;" ::"n"(kShareRing - 1) : "memory");
        state.take(ring0 + (uint32_t)(st % kShareRing) * kDecStepBytes, here.row + hw, here.row1, scale_log2);
        const Walk done = here;
        const bool other = next_step(here, batch, n_q_heads);
        if (!other && here.left > 0) continue;
        // ---- end of a part: combined like a split of decode_kernel.  One barrier: a warp that is a part ahead
        // writes to the other buffer.
        DecShared<1>& sh = shared_parts[part & 1];
        state.leave(sh, warp, lane, scale_log2);
        __syncthreads();
        if (threadIdx.x < kHeadDim) {
            const int t = threadIdx.x;
            const DecodeReq& rq = batch.r[done.r];
            float mx, lsum, osum;
            add_warps(sh, 0, t, scale_log2, mx, lsum, osum);
            if (from_start && done.row1 == rq.len + 1) {
                out[((long long)rq.index * n_q_heads + done.h) * kHeadDim + t] = osum / lsum;
            } else {
                float* rec = parts + (2ll * blockIdx.x + (part > 0)) * (kHeadDim + 2);
                if (t == 0) { rec[0] = mx; rec[1] = lsum; }
                rec[2 + t] = osum;
            }
        }
        ++part;
        if (other) begin_part();
        from_start = true;
    }
}

// ---------------------------------------------------------------------------------------------
// Grouped queries: several query heads attend over the same rows.  With the scalar kernel above the
// arithmetic (four shuffles and sixteen FMAs per lane, row and head) takes longer than the rows take
// to arrive, so this one multiplies on the tensor cores (mma.sync m16n8k16; per row it is a
// bandwidth-bound kernel, far from needing tcgen05's rate):
//   S = Q K^T   A = query heads, B = sixteen key rows;  O += P V   A = probabilities, B = value rows.
// The sixteen rows of A hold the GP <= 8 heads of the pass several times over.  In S the copies are
// equal; in P they are the three bf16 terms of the fp32 probability (24 bits together), so that the
// product keeps the precision of fp32 probabilities: row r belongs to head r mod GP and term r / GP.
// With GP = 8 only two terms fit and a second product adds the third.
// A CTA of four warps takes a split; a warp takes sixteen rows of K and V at a time through a
// cp.async ring of its own, 16-byte chunks XOR-swizzled so that ldmatrix is free of bank conflicts.
// The reference of the running softmax moves only when a logit leaves it by 2^8.
// ---------------------------------------------------------------------------------------------
constexpr int kMmaThreads = 128;
constexpr int kMmaWarps = kMmaThreads / 32;
constexpr int kMmaRows = 16;                         // rows per warp and step
constexpr int kMmaRing = 3;                          // steps in a warp's ring (all but one in flight)
constexpr int kMmaStepBytes = 2 * kMmaRows * kDecRowBytes;         // [K|V][row][256 B]
constexpr int kMmaRingBytes = kMmaWarps * kMmaRing * kMmaStepBytes;
static_assert(kMmaRingBytes * (kDecodeMaxCtasPerSm + 1) > (228 << 10) && kDecRingBytes * (kDecodeMaxCtasPerSm + 1) > (228 << 10),
              "the workspace has room for the splits of kDecodeMaxCtasPerSm CTAs per SM");
constexpr float kMmaSlack = 8.f;                     // log2 by which a logit may exceed the reference

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&b);
}
// Terms `part` (0, 1, 2; else zero) of the bf16 expansions of two fp32 values.
__device__ __forceinline__ uint32_t bf16_term(float x, float y, int part) {
    if (part >= 1) { x -= __bfloat162float(__float2bfloat16_rn(x)); y -= __bfloat162float(__float2bfloat16_rn(y)); }
    if (part >= 2) { x -= __bfloat162float(__float2bfloat16_rn(x)); y -= __bfloat162float(__float2bfloat16_rn(y)); }
    return part >= 3 ? 0u : pack_bf16(x, y);
}

template <int GP>
struct MmaShared {
    float m[kMmaWarps][GP];
    float l[kMmaWarps][GP];
    float o[kMmaWarps][GP][kHeadDim];
};

// gt <= GP query heads of the group are handled per pass over the rows.
template <class Batch, int GP, bool kClustered>
__global__ void __launch_bounds__(kMmaThreads)
decode_mma_kernel(const __grid_constant__ Batch batch, const __nv_bfloat16* __restrict__ q,
                  const __nv_bfloat16* __restrict__ k_new, const __nv_bfloat16* __restrict__ v_new,
                  __nv_bfloat16* __restrict__ cache_k, __nv_bfloat16* __restrict__ cache_v,
                  long long stride_row, long long stride_head, int n_q_heads, int n_kv_heads, int group, int gt,
                  int rows_per_split, float scale_log2, float* __restrict__ parts, float* __restrict__ out) {
    __shared__ MmaShared<GP> sh;
    __shared__ ClusterShared<GP> cs;
    extern __shared__ __align__(128) uint8_t dec_ring[];         // [warp][ring step][K|V][row][256 B, swizzled]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int r = 0;
    {
        int lo = 0, hi = batch.n_req - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (batch.r[mid].cta_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        r = lo;
    }
    const DecodeReq rq = batch.r[r];
    const int n_pass = group / gt;
    const int local = (int)blockIdx.x - rq.cta_begin;            // [head][pass][split]
    const int split = local % rq.n_splits;
    const int pass = (local / rq.n_splits) % n_pass;
    const int h = local / (rq.n_splits * n_pass);
    const int n_rows = rq.len + 1;                               // cached rows + the new one
    const int row0 = split * rows_per_split, row1 = min(n_rows, row0 + rows_per_split);
    const int qh0 = h * group + pass * gt;                       // first query head of this pass

    prefetch_rows(cache_k, cache_v, (rq.begin + row0) * stride_row + h * stride_head, stride_row, min(row1, rq.len) - row0);
    grid_dependency_wait();

    const long long head_off = (long long)h * stride_head;
    const __nv_bfloat16* ck = cache_k + rq.begin * stride_row + head_off;
    const __nv_bfloat16* cv = cache_v + rq.begin * stride_row + head_off;
    const __nv_bfloat16* nk = k_new + ((long long)rq.index * n_kv_heads + h) * kHeadDim;
    const __nv_bfloat16* nv = v_new + ((long long)rq.index * n_kv_heads + h) * kHeadDim;

    // Copies of one step: half a warp per row, 16 bytes per lane; rows past the split are zero-filled
    // (and masked below).  Chunk c of row i goes to chunk c xor (i mod 8).
    const int l16 = lane & 15, hi_half = lane >> 4;
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(dec_ring) + warp * (kMmaRing * kMmaStepBytes);
    auto issue = [&](int step) {
        const int base = row0 + (step * kMmaWarps + warp) * kMmaRows;
        const uint32_t dst = ring0 + (uint32_t)(step % kMmaRing) * kMmaStepBytes;
        if (base < row1) {
#pragma unroll
            for (int f = 0; f < kMmaRows / 2; ++f) {
                const int i = 2 * f + hi_half;
                const int row = base + i;
                const bool is_new = (row == rq.len);
                const bool valid = row < row1;
                const __nv_bfloat16* kp = ((is_new || !valid) ? nk : ck + (long long)row * stride_row) + l16 * 8;
                const __nv_bfloat16* vp = ((is_new || !valid) ? nv : cv + (long long)row * stride_row) + l16 * 8;
                const int nbytes = valid ? 16 : 0;
                const uint32_t at = dst + i * kDecRowBytes + ((l16 ^ (i & 7)) << 4);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(at), "l"(kp), "r"(nbytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                             ::"r"(at + kMmaRows * kDecRowBytes), "l"(vp), "r"(nbytes) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int n_groups = (row1 - row0 + kMmaRows - 1) / kMmaRows;                // of sixteen rows in the split
    const int n_steps = n_groups > warp ? (n_groups - warp + kMmaWarps - 1) / kMmaWarps : 0;
#pragma unroll
    for (int st = 0; st < kMmaRing - 1; ++st) issue(st);

    // Query fragments: A row lane / 4 (and + 8, which is the same head) is head (lane / 4) mod GP.
    const int head = (lane >> 2) % GP;
    const int part_lo = (lane >> 2) / GP, part_hi = ((lane >> 2) + 8) / GP;      // terms of this lane's two rows of P
    uint32_t qa[8][2];
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
        const __nv_bfloat16* src = q + ((long long)rq.index * n_q_heads + qh0 + head) * kHeadDim + kk * 16 + (lane & 3) * 2;
        qa[kk][0] = head < gt ? *reinterpret_cast<const uint32_t*>(src) : 0u;
        qa[kk][1] = head < gt ? *reinterpret_cast<const uint32_t*>(src + 8) : 0u;
    }
    // The appended row (Eq. 2) is also written into the cache by the CTA that owns it on the group's
    // first pass (nobody reads cache row `len` in this step).
    if (pass == 0 && rq.len >= row0 && rq.len < row1 && warp == 0) {
        const __nv_bfloat16* src = (lane < 16 ? nk : nv) + l16 * 8;
        __nv_bfloat16* dst = (lane < 16 ? cache_k : cache_v) + rq.begin * stride_row + head_off +
                             (long long)rq.len * stride_row + l16 * 8;
        *reinterpret_cast<uint4*>(dst) = __ldg(reinterpret_cast<const uint4*>(src));
    }

    float o[16][4];                                  // feature group j: features 8j + 2 (lane mod 4), + 1; rows lane / 4, + 8
#pragma unroll
    for (int j = 0; j < 16; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[j][c] = 0.f;
    // Reference (in units of the raw product, like the scalar kernel's) and sum (over this lane's keys) of the
    // head.  The reference starts finite, so that logits of -inf met before any other count nothing.
    float m = -FLT_MAX, l = 0.f;
    // ldmatrix: matrix i of an x4 is addressed by lanes 8i .. 8i + 7
    const int mi = lane >> 3, mr = lane & 7;
    const int k_row = (mi >> 1) * 8 + mr, k_chunk = mi & 1;      // K: (rows 0-7, 8-15) x (chunk, next chunk)
    const int v_row = (mi & 1) * 8 + mr, v_chunk = mi >> 1;      // V: two row halves of one chunk, then of the next

    for (int st = 0; st < n_steps; ++st) {
        issue(st + kMmaRing - 1);                    // into the buffer that was consumed one iteration ago
        asm volatile("cp.async.wait_group %0;" ::"n"(kMmaRing - 1) : "memory");
        __syncwarp();                                // every lane's copies are visible to the whole warp
        const int base = row0 + (st * kMmaWarps + warp) * kMmaRows;
        const uint32_t kbuf = ring0 + (uint32_t)(st % kMmaRing) * kMmaStepBytes;
        const uint32_t vbuf = kbuf + kMmaRows * kDecRowBytes;
        // this lane's four products: keys 2 (lane mod 4), + 1 of keys 0-7 and of 8-15 (rows + 8 are copies);
        // sums over sixteen features, added pair by pair in fp32 (see below)
        float x[4], part[3][4];
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            uint32_t b[4];
            ldmatrix_x4(b, kbuf + k_row * kDecRowBytes + (((2 * kk + k_chunk) ^ (k_row & 7)) << 4));
            float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(s0, qa[kk][0], qa[kk][0], qa[kk][1], qa[kk][1], b[0], b[1]);
            mma_bf16(s1, qa[kk][0], qa[kk][0], qa[kk][1], qa[kk][1], b[2], b[3]);
            const float now[4] = {s0[0], s0[1], s1[0], s1[1]};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                x[c] = now[c];
                if (kk & 1) x[c] += part[0][c]; else part[0][c] = x[c];
                if ((kk & 3) == 3) x[c] += part[1][c]; else if ((kk & 3) == 1) part[1][c] = x[c];
                if (kk == 7) x[c] += part[2][c]; else if (kk == 3) part[2][c] = x[c];
            }
        }
        if (base + kMmaRows > row1) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (base + (i >> 1) * 8 + (lane & 3) * 2 + (i & 1) >= row1) x[i] = -INFINITY;
        }
        float mx = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        float alpha = 1.f;
        if (__any_sync(0xffffffffu, (mx - m) * scale_log2 > kMmaSlack)) {      // also the first step
            const float to = fmaxf(m, mx);
            alpha = dec_ex2((m - to) * scale_log2);
            m = to;
            l *= alpha;
        }
        float pr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { pr[i] = dec_ex2((x[i] - m) * scale_log2); l += pr[i]; }
        const uint32_t a0 = bf16_term(pr[0], pr[1], part_lo), a1 = bf16_term(pr[0], pr[1], part_hi);
        const uint32_t a2 = bf16_term(pr[2], pr[3], part_lo), a3 = bf16_term(pr[2], pr[3], part_hi);
        const uint32_t c0 = GP == 8 ? bf16_term(pr[0], pr[1], 2) : 0u, c2 = GP == 8 ? bf16_term(pr[2], pr[3], 2) : 0u;
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            uint32_t b[4];
            ldmatrix_x4_trans(b, vbuf + v_row * kDecRowBytes + (((j + v_chunk) ^ (v_row & 7)) << 4));
            // the step's sums start from zero and are added in fp32: the tensor core truncates what it adds
            // to, which over a long cache would show (30000 rows, 8 heads per row: 5.8e-7 against 2.6e-7)
            float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(t0, a0, a1, a2, a3, b[0], b[1]);
            mma_bf16(t1, a0, a1, a2, a3, b[2], b[3]);
            if (GP == 8) {                           // (rows 0-7 of this product are zeros: only rows 8-15 are taken)
                float u0[4] = {0.f, 0.f, 0.f, 0.f}, u1[4] = {0.f, 0.f, 0.f, 0.f};
                mma_bf16(u0, 0u, c0, 0u, c2, b[0], b[1]);
                mma_bf16(u1, 0u, c0, 0u, c2, b[2], b[3]);
                t0[2] += u0[2], t0[3] += u0[3];
                t1[2] += u1[2], t1[3] += u1[3];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                o[j][c] = fmaf(o[j][c], alpha, t0[c]);
                o[j + 1][c] = fmaf(o[j + 1][c], alpha, t1[c]);
            }
        }
        __syncwarp();                                // the buffer may be refilled
    }

    // ---- combine: the terms of a head in registers, then the warps in warp order -----------------
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    // The first term of a probability takes part on its own, the sum of the others is a correction: with
    // an infinite value the first term's sum is the result (the others may be zero times infinity).
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float y[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float low = (part_lo > 0 && part_lo < 3 ? o[j][c] : 0.f) + (part_hi < 3 ? o[j][c + 2] : 0.f);
#pragma unroll
            for (int ofs = 16; ofs >= 4 * GP; ofs >>= 1) low += __shfl_xor_sync(0xffffffffu, low, ofs);      // rows lane / 4 of the same head
            y[c] = isinf(o[j][c]) ? o[j][c] : o[j][c] + low;
        }
        if (part_lo == 0) {
            sh.o[warp][head][8 * j + 2 * (lane & 3)] = y[0];
            sh.o[warp][head][8 * j + 2 * (lane & 3) + 1] = y[1];
        }
    }
    if (part_lo == 0 && (lane & 3) == 0) { sh.m[warp][head] = m; sh.l[warp][head] = l; }
    __syncthreads();
    // thread t owns feature t of every query head of the pass
    const int n_splits = rq.n_splits;
    const long long part_stride = kHeadDim + 2;                  // m, l, o[128]
    float* my_parts = parts + ((long long)rq.part_begin + ((long long)(h * n_pass + pass) * n_splits + split) * gt) * part_stride;
    const int t = threadIdx.x;
    for (int g = 0; g < gt; ++g) {
        float mx = -INFINITY;
#pragma unroll
        for (int w = 0; w < kMmaWarps; ++w) mx = fmaxf(mx, sh.m[w][g]);
        float lsum = 0.f, osum = 0.f;
#pragma unroll
        for (int w = 0; w < kMmaWarps; ++w) {
            const float a = dec_ex2((sh.m[w][g] - mx) * scale_log2);             // (an idle warp's sums are 0)
            lsum = fmaf(sh.l[w][g], a, lsum);
            osum = fmaf(sh.o[w][g][t], a, osum);
        }
        if (kClustered) {
            if (t == 0) { cs.m[g] = mx; cs.l[g] = lsum; }
            cs.o[g][t] = osum;
        } else if (n_splits == 1) {
            out[((long long)rq.index * n_q_heads + qh0 + g) * kHeadDim + t] = osum / lsum;
        } else {
            float* rec = my_parts + g * part_stride;
            if (t == 0) { rec[0] = mx; rec[1] = lsum; }
            rec[2 + t] = osum;
        }
    }
    if (kClustered) cluster_combine(cs, n_splits, gt, scale_log2, out + ((long long)rq.index * n_q_heads + qh0) * kHeadDim);
}

// Several splits: adds the partial results of one (request, KV head, pass, query head) in split
// order.  One CTA of 128 threads per such unit, thread t owns feature t; the splits' reference
// values are fetched in one round trip and the records of sixteen splits are requested together
// (the kernel is bound by the latency of these loads).  Launched
// behind decode_kernel with programmatic stream serialisation: no counters, no atomics, nothing in
// the workspace has to be cleared, and the order of additions is fixed.
template <class Batch>
__global__ void __launch_bounds__(kHeadDim)
decode_combine_kernel(const __grid_constant__ Batch batch, int gt, int n_pass, int n_q_heads, int group,
                      float scale_log2, const float* __restrict__ parts, float* __restrict__ out) {
    const DecodeReq rq = batch.r[blockIdx.y];
    const int g = (int)blockIdx.x % gt, unit = (int)blockIdx.x / gt;     // unit = h * n_pass + pass
    const int pass = unit % n_pass, h = unit / n_pass;
    const int t = threadIdx.x;
    const long long part_stride = kHeadDim + 2;
    int n_splits;                                                // partial results of the unit,
    const float* base;                                           // the first of them (but see `skip`),
    long long step, skip = 0;                                    // and from one to the next
    if (batch.share > 0) {
        // the CTAs whose shares hold the unit's first and last step.  The unit is the first CTA's last one, in
        // its second record, unless the share begins with it; it is the others' first.
        const int steps = unit_steps(rq);
        const long long s0 = rq.step_begin + (long long)unit * steps;
        const int c0 = share_of(batch, s0);
        n_splits = share_of(batch, s0 + steps - 1) - c0 + 1;
        base = parts + 2ll * c0 * part_stride;
        step = 2 * part_stride;
        skip = share_begin(batch, c0) == s0 ? 0 : part_stride;
    } else {
        n_splits = rq.n_splits;
        base = parts + (rq.part_begin + (long long)unit * n_splits * gt + g) * part_stride;
        step = (long long)gt * part_stride;
    }
    grid_dependency_wait();
    if (n_splits == 1) return;                                   // the output is already written
    const auto record = [&](int i) { return base + i * step + (i == 0 ? skip : 0); };
    // largest reference value over the splits: thread t looks at splits t, t + 128, ...; one round
    // trip for up to 128 splits, then a block-wide maximum
    __shared__ float warp_max[kHeadDim / 32];
    float mx = -INFINITY;
    for (int sp = t; sp < n_splits; sp += kHeadDim) mx = fmaxf(mx, __ldcg(record(sp)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((t & 31) == 0) warp_max[t >> 5] = mx;
    __syncthreads();
    mx = fmaxf(fmaxf(warp_max[0], warp_max[1]), fmaxf(warp_max[2], warp_max[3]));
    // the records in split order, kBatch of them requested together
    constexpr int kBatch = 16;
    float lsum = 0.f, osum = 0.f;
    for (int s0 = 0; s0 < n_splits; s0 += kBatch) {
        float mv[kBatch], lv[kBatch], ov[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const bool in = s0 + j < n_splits;
            const float* rec = record(s0 + j);
            mv[j] = in ? __ldcg(rec) : -INFINITY;
            lv[j] = in ? __ldcg(rec + 1) : 0.f;
            ov[j] = in ? __ldcg(rec + 2 + t) : 0.f;
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const float a = dec_ex2((mv[j] - mx) * scale_log2);  // 0 past the last split
            lsum = fmaf(lv[j], a, lsum);
            osum = fmaf(ov[j], a, osum);
        }
    }
    out[((long long)rq.index * n_q_heads + h * group + pass * gt + g) * kHeadDim + t] = osum / lsum;
}

}  // namespace

namespace {

template <class Batch>
struct Kernels {
    typedef void (*Scalar)(Batch, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*,
                           __nv_bfloat16*, long long, long long, int, int, int, int, float, float*, float*);
    typedef void (*Mma)(Batch, const __nv_bfloat16*, const __nv_bfloat16*, const __nv_bfloat16*, __nv_bfloat16*,
                        __nv_bfloat16*, long long, long long, int, int, int, int, int, float, float*, float*);
    static Scalar scalar(int gt, bool clustered) {
        return gt == 2 ? (clustered ? decode_kernel<Batch, 2, true> : decode_kernel<Batch, 2, false>)
                       : (clustered ? decode_kernel<Batch, 1, true> : decode_kernel<Batch, 1, false>);
    }
    static Mma mma(int gt, bool clustered) {
        if (clustered)
            return gt > 4 ? decode_mma_kernel<Batch, 8, true> : gt > 2 ? decode_mma_kernel<Batch, 4, true> : decode_mma_kernel<Batch, 2, true>;
        return gt > 4 ? decode_mma_kernel<Batch, 8, false> : gt > 2 ? decode_mma_kernel<Batch, 4, false> : decode_mma_kernel<Batch, 2, false>;
    }
    static cudaError_t configure() {
        cudaError_t e = cudaFuncSetAttribute(decode_shared_kernel<Batch>, cudaFuncAttributeMaxDynamicSharedMemorySize, kShareRingBytes);
        for (bool clustered : {false, true}) {
            for (int gt : {1, 2})
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(scalar(gt, clustered), cudaFuncAttributeMaxDynamicSharedMemorySize, kDecRingBytes);
            for (int gt : {2, 4, 8})
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(mma(gt, clustered), cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaRingBytes);
        }
        return e;
    }
};

// The rings need more dynamic shared memory than the default limit: raised once per device.
cudaError_t configure_decode() {
    static unsigned long long configured = 0;
    return once_per_device(configured, []() {
        cudaError_t e = Kernels<DecodeBatch>::configure();
        if (e == cudaSuccess) e = Kernels<DecodeBatchOf<1>>::configure();
        return e != cudaSuccess ? e : Kernels<DecodeBatchOf<kDecodeFew>>::configure();
    });
}

// f(batch), in the smallest argument that holds its requests
template <int kRequests, class F>
cudaError_t with_copy(const DecodeBatch& batch, F f) {
    DecodeBatchOf<kRequests> few;
    few.n_req = batch.n_req;
    few.share = batch.share;
    few.longer = batch.longer;
    few.pad = 0;
    for (int i = 0; i < kRequests; ++i) few.r[i] = batch.r[i];          // (those past the last are zeros)
    return f(few);
}
template <class F>
cudaError_t with_batch(const DecodeBatch& batch, F f) {
    return batch.n_req == 1 ? with_copy<1>(batch, f) : batch.n_req <= kDecodeFew ? with_copy<kDecodeFew>(batch, f) : f(batch);
}

}  // namespace

// CTAs that one SM holds at a time of the kernel that handles gt query heads per pass, on the current
// device (looked up once per device); 0 if the query fails.  The planner sizes the grid to one wave.
int decode_ctas_per_sm(int gt, bool mma) {
    static int cache[64][5] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    const int idx = !mma ? gt - 1 : gt > 4 ? 4 : gt > 2 ? 3 : 2;
    int v = __atomic_load_n(&cache[dev][idx], __ATOMIC_ACQUIRE);
    if (v > 0) return v;
    if (configure_decode() != cudaSuccess) { cudaGetLastError(); return 0; }
    typedef Kernels<DecodeBatch> K;
    const cudaError_t err = mma ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, K::mma(gt, false), kMmaThreads, kMmaRingBytes)
                                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, K::scalar(gt, false), kDecThreads, kDecRingBytes);
    if (err != cudaSuccess || v <= 0) { cudaGetLastError(); return 0; }
    __atomic_store_n(&cache[dev][idx], v, __ATOMIC_RELEASE);
    return v;
}

cudaError_t launch_decode(const DecodeBatch& all, int total_ctas, int gt, bool mma, int cluster, const void* q,
                          const void* k_new, const void* v_new, void* cache_k, void* cache_v,
                          long long stride_row, long long stride_head, int n_q_heads, int n_kv_heads,
                          int rows_per_split, float scale_log2, float* parts, float* out,
                          cudaStream_t stream) {
    if (total_ctas <= 0) return cudaSuccess;
    const int group = n_q_heads / n_kv_heads;
    cudaError_t err = configure_decode();
    if (err != cudaSuccess) return err;
    const bool clustered = cluster > 1;
    const dim3 grid((unsigned)total_ctas);
    const auto *qb = (const __nv_bfloat16*)q, *kb = (const __nv_bfloat16*)k_new, *vb = (const __nv_bfloat16*)v_new;
    auto *ck = (__nv_bfloat16*)cache_k, *cv = (__nv_bfloat16*)cache_v;
    return with_batch(all, [&](const auto& batch) {
        typedef Kernels<typename std::decay<decltype(batch)>::type> K;
        typedef typename std::decay<decltype(batch)>::type Batch;
        if (batch.share > 0)
            return launch_chained(decode_shared_kernel<Batch>, grid, dim3(kDecThreads), (size_t)kShareRingBytes, stream, batch, qb, kb, vb,
                                  ck, cv, stride_row, stride_head, n_q_heads, n_kv_heads, group, scale_log2, parts, out);
        if (mma)
            return launch_chained_clusters(K::mma(gt, clustered), grid, dim3(kMmaThreads), (unsigned)cluster, (size_t)kMmaRingBytes, stream,
                                           batch, qb, kb, vb, ck, cv, stride_row, stride_head, n_q_heads, n_kv_heads, group, gt,
                                           rows_per_split, scale_log2, parts, out);
        return launch_chained_clusters(K::scalar(gt, clustered), grid, dim3(kDecThreads), (unsigned)cluster, (size_t)kDecRingBytes, stream,
                                       batch, qb, kb, vb, ck, cv, stride_row, stride_head, n_q_heads, n_kv_heads, group, rows_per_split,
                                       scale_log2, parts, out);
    });
}

cudaError_t launch_decode_combine(const DecodeBatch& all, int gt, int n_q_heads, int n_kv_heads,
                                  float scale_log2, const float* parts, float* out, cudaStream_t stream) {
    const int group = n_q_heads / n_kv_heads;
    const int n_pass = group / gt;
    return with_batch(all, [&](const auto& batch) {
        return launch_chained(decode_combine_kernel<typename std::decay<decltype(batch)>::type>,
                              dim3((unsigned)(n_kv_heads * n_pass * gt), (unsigned)batch.n_req), dim3(kHeadDim), 0, stream, batch, gt,
                              n_pass, n_q_heads, group, scale_log2, parts, out);
    });
}

}  // namespace lookm
