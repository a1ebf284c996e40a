// Bandwidth-bound kernels of the path: key norms, compaction of the kept keys (the B operand of
// the matching), row arg-max of given similarity matrices, inversion of the evicted->kept
// assignment into per-kept-row member lists, and the merge/compact kernel (Eq. 6-7, 10-12).
//
// A K or V row is 128 bf16 = 256 bytes = 16 lanes x 16 bytes, so a half-warp moves one row with
// one 16-byte access per lane.
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"

namespace lookm {
namespace {

struct Row8 { float v[8]; };

__device__ __forceinline__ Row8 unpack8(const uint4& u) {
    Row8 r;
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        r.v[2 * i] = __uint_as_float(w[i] << 16);
        r.v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
    return r;
}

__device__ __forceinline__ uint4 pack8(const Row8& r) {
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(r.v[2 * i], r.v[2 * i + 1]);
        w[i] = *reinterpret_cast<const unsigned*>(&b);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// A request to shared memory, by the first threads of the CTA.
__device__ __forceinline__ void copy_words(Req& to, const Req& from) {
    if (threadIdx.x < sizeof(Req) / 4) reinterpret_cast<int*>(&to)[threadIdx.x] = reinterpret_cast<const int*>(&from)[threadIdx.x];
}
__device__ __forceinline__ Req find_req_by_slot(const ReqTable& reqs, long long g) {
    if (reqs.n == 1) return reqs.only;
    int lo = 0, hi = reqs.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long long)reqs.rows[mid].slot_begin <= g) lo = mid; else hi = mid - 1;
    }
    return reqs.rows[lo];
}

// ---------------------------------------------------------------------------------------------
// 1 / |k| of every key row (0 for a zero row), the cosine denominators of Eq. 9.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
key_norms_kernel(const __nv_bfloat16* __restrict__ k, long long stride_tok, long long stride_head,
                 int n_kv_heads, long long T, float* __restrict__ rnorm_all) {
    const int half = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const long long n_rows = T * n_kv_heads;
    // the loop bound is the warp's first row, so that both half-warps always reach the shuffles
    for (long long rw = (long long)blockIdx.x * 16 + (half & ~1); rw < n_rows; rw += (long long)gridDim.x * 16) {
        const long long r = rw + (half & 1);
        const bool valid = r < n_rows;
        const long long tok = valid ? r / n_kv_heads : 0;
        const int h = valid ? (int)(r % n_kv_heads) : 0;
        const uint4 u = *reinterpret_cast<const uint4*>(k + tok * stride_tok + h * stride_head + l16 * 8);
        const Row8 x = unpack8(u);
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) ss = fmaf(x.v[i], x.v[i], ss);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o, 16);
        if (l16 == 0 && valid) rnorm_all[(long long)h * T + tok] = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
    }
}

// ---------------------------------------------------------------------------------------------
// Kept keys of every (request, head) copied into one dense [rows, 128] matrix in kept-list
// order, with their inverse norms.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
gather_kept_kernel(const __nv_bfloat16* __restrict__ k, long long stride_tok, long long stride_head,
                   const __grid_constant__ ReqTable reqs, int n_kv_heads, long long T,
                   long long total_rows, const int* __restrict__ kept_idx,
                   const float* __restrict__ rnorm_all, __nv_bfloat16* __restrict__ kept_keys,
                   float* __restrict__ rnorm_kept, int* status) {
    grid_dependency_wait();
    const int half = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const long long g = (long long)blockIdx.x * 16 + half;
    if (g >= total_rows) return;
    const Req rq = find_req_by_slot(reqs, g);
    if (rq.mode == LOOKM_MERGE_NONE) return;             // nothing is matched against its kept keys
    const int u = (int)(g - rq.slot_begin);              // (there are fewer than 2^31 kept rows in all)
    const int h = u / rq.B;
    const long long dst = rq.kept_off + u;
    int pos = kept_idx[dst];
    if (pos < 0 || pos >= rq.L) { if (l16 == 0) atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pos = 0; }
    const long long tok = rq.tok_begin + pos;
    const uint4 u4 = *reinterpret_cast<const uint4*>(k + tok * stride_tok + h * stride_head + l16 * 8);
    *reinterpret_cast<uint4*>(kept_keys + dst * kHeadDim + l16 * 8) = u4;
    if (l16 == 0) rnorm_kept[dst] = rnorm_all[(long long)h * T + tok];
}

// ---------------------------------------------------------------------------------------------
// Eviction alone (Eq. 6-7): kept K and V rows of the requests with LOOKM_MERGE_NONE copied to the
// output cache, one warp per row (lanes 0-15 the K row, 16-31 the V row).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
compact_kept_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                    long long stride_tok, long long stride_head, const __grid_constant__ ReqTable reqs,
                    int n_kv_heads, long long total_rows, const int* __restrict__ kept_idx,
                    int varlen_output, long long out_stride_head, __nv_bfloat16* __restrict__ out_k,
                    __nv_bfloat16* __restrict__ out_v, int* status) {
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, l16 = lane & 15;
    const long long g = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (g >= total_rows) return;
    const Req rq = find_req_by_slot(reqs, g);
    if (rq.mode != LOOKM_MERGE_NONE) return;
    const long long u = g - rq.slot_begin;
    const int h = (int)(u / rq.B), slot = (int)(u % rq.B);
    int pos = kept_idx[rq.kept_off + (long long)h * rq.B + slot];
    if (pos < 0 || pos >= rq.L) { if (lane == 0) atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pos = 0; }
    const __nv_bfloat16* src = (lane < 16 ? k : v) + (rq.tok_begin + (long long)pos) * stride_tok +
                               (long long)h * stride_head + l16 * 8;
    long long dst;
    if (varlen_output) dst = (((long long)rq.out_begin + slot) * n_kv_heads + h) * kHeadDim;
    else dst = (long long)h * out_stride_head + (long long)slot * kHeadDim;
    *reinterpret_cast<uint4*>((lane < 16 ? out_k : out_v) + dst + l16 * 8) = *reinterpret_cast<const uint4*>(src);
}

// ---------------------------------------------------------------------------------------------
// Row arg-max of given similarity blocks (one warp per evicted row); lowest slot wins ties.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
argmax_rows_kernel(const float* __restrict__ sim_matrix, const __grid_constant__ ReqTable reqs,
                   int n_kv_heads, int* __restrict__ assign, float* __restrict__ sim) {
    const Req rq = reqs.get(blockIdx.z);
    const int h = blockIdx.y;
    const int e = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= rq.E) return;
    const float* row = sim_matrix + rq.sim_off + ((long long)h * rq.E + e) * rq.B;
    float best = -INFINITY;
    int slot = 0x7fffffff;
    for (int c = lane; c < rq.B; c += 32) {
        const float v = row[c];
        if (v > best) { best = v; slot = c; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int os = __shfl_xor_sync(0xffffffffu, slot, o);
        if (ob > best || (ob == best && os < slot)) { best = ob; slot = os; }
    }
    if (lane == 0) {
        assign[rq.ev_off + (long long)h * rq.E + e] = slot;
        sim[rq.ev_off + (long long)h * rq.E + e] = best;
    }
}

// ---------------------------------------------------------------------------------------------
// Inversion of the assignment: for each (request, head) a stable sort of the evicted ranks by
// their kept slot gives, per kept row, its members in ascending position; the result is the merge
// kernel's entry list (position and weight of every kept row and, behind it, of its members).  A cluster
// of CTAs per (request, head); stable LSD radix sort: every warp of the cluster owns a contiguous segment of the
// list, ranks equal digits inside a 32-element step with ballots, and adds the counts of earlier steps,
// of earlier warps and, read from their shared memory, of earlier CTAs.
// What bounds it is the chain of dependent steps, not the bytes: a list of 26214 evicted tokens is 100
// KB.  One CTA of 32 warps per list | up to eight of 16: 26214 evicted tokens x 8 heads into 6554 slots
// 164 | 43 us, 13107 x 40 into 3277 92 | 46, 7388 x 8 into 389 22 | 16.
// ---------------------------------------------------------------------------------------------
constexpr int kInvThreads = 512;
constexpr int kInvWarps = kInvThreads / 32;
constexpr int kInvBatch = 8;                         // loop steps whose loads are issued together

// Second half of the entry list: the kept rows (flagged with the sign bit, weight = member count),
// for every work unit (unit u of a head covers the entries [u * unit_entries, (u + 1) * unit_entries))
// the slot its first entry belongs to, with that slot's first entry and member count, and a
// cleared arrival counter per slot.  Slot c, whose kept row is at position pc, has n members, after
// those of the slots before it.
struct KeptEntries {
    int2* ent;                                           // position and weight
    int4* units;                                         // [unit of the head][head]
    int* slot_cnt;
    int* status;
    int L, unit_entries, h, n_kv_heads;
    __device__ __forceinline__ void write(int c, int pc, int begin, int n) const {
        if (pc < 0 || pc >= L) { atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pc = 0; }
        const int s_c = c + begin;                       // entry of the kept row
        const int s_next = s_c + n + 1;                  // entry of the next kept row (L after the last)
        ent[s_c] = make_int2(pc | (int)0x80000000, __float_as_int((float)n));
        slot_cnt[c] = 0;
        for (int u = (s_c + unit_entries - 1) / unit_entries; u * unit_entries < s_next; ++u)
            units[(long long)u * n_kv_heads + h] = make_int4(c, s_c, n, 0);
    }
};

// Lanes of the warp that hold a valid element with the same digit as the caller: one ballot per
// digit bit (match.any takes a step per distinct value, i.e. up to 32 for well-mixed digits).
template <int kMaxBits>
__device__ __forceinline__ unsigned same_digit_lanes(unsigned d, bool valid, int dbits) {
    unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < kMaxBits; ++b) {
        if (b < dbits) {
            const bool bit = (d >> b) & 1u;
            const unsigned bal = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bal : ~bal;
        }
    }
    return peers;
}

// CountT / kMaxBits: 16-bit counters with digits of up to 11 bits when no request of the call evicts
// more than 65535 tokens per head (every count and prefix then fits), else 32-bit counters with
// digits of up to 10 bits.
template <typename CountT, int kMaxBits>
__global__ void __launch_bounds__(kInvThreads, 2)
invert_assignment_kernel(const int* __restrict__ assign, const int* __restrict__ kept_idx,
                         const int* __restrict__ evict_idx,
                         const float* __restrict__ sim, const __grid_constant__ ReqTable reqs,
                         int n_kv_heads, int ctas, long long T, int* row_begin,
                         int2* __restrict__ entries,
                         int4* __restrict__ unit_first, int* __restrict__ slot_cnt,
                         unsigned* sort_a, unsigned* sort_b, int* status) {
    static_assert((1 << kMaxBits) <= 4 * kInvThreads, "a thread scans four digits");
    extern __shared__ __align__(16) unsigned char inv_smem[];
    __shared__ int warp_sums[kInvWarps];
    grid_dependency_wait();
    const Req rq = reqs.get(blockIdx.y);
    if (rq.mode == LOOKM_MERGE_NONE) return;             // its kept rows are copied, nothing is merged
    const int h = blockIdx.x / ctas, cta = blockIdx.x % ctas;     // the cluster: the CTAs of one head
    const int E = rq.E, B = rq.B;
    const long long ev_base = rq.ev_off + (long long)h * E;
    int* rp = row_begin + rq.rp_off + (long long)h * (B + 1);     // scratch of several passes: first member of a slot
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int thread = cta * kInvThreads + threadIdx.x, n_threads = ctas * kInvThreads;   // of the cluster
    auto sync = [&]() { if (ctas > 1) ptx::cluster_sync(); else __syncthreads(); };

    // entry list of this (request, head): for every kept slot its kept row, then its members
    int2* ent = entries + (long long)h * T + rq.tok_begin;
    const KeptEntries kept = {ent, unit_first + rq.unit_begin, slot_cnt + rq.kept_off + (long long)h * B, status,
                              rq.L, rq.unit_entries, h, n_kv_heads};
    const int* kept_idx_head = kept_idx + rq.kept_off + (long long)h * B;
    const bool weighted = (rq.mode == LOOKM_MERGE_WEIGHTED);
    if (E == 0) {
        for (int c = thread; c < B; c += n_threads) kept.write(c, kept_idx_head[c], 0, 0);
        return;
    }
    // segment of the list owned by each warp: a multiple of 32 elements
    const int n_warps = ctas * kInvWarps;
    const int seg = ((E + n_warps * 32 - 1) / (n_warps * 32)) * 32;
    const int s_begin = (int)min((long long)E, (long long)(cta * kInvWarps + warp) * seg), s_end = min(E, s_begin + seg);

    int n_pass, dbits;
    invert_digits(B, kMaxBits, n_pass, dbits);
    const int nd = 1 << dbits;
    const unsigned dmask = (unsigned)nd - 1u;
    const int padded = max(nd, 4);
    CountT* cnt = reinterpret_cast<CountT*>(inv_smem);                          // [warp][digit]
    int* digit_tot = reinterpret_cast<int*>(inv_smem + (size_t)kInvWarps * padded * sizeof(CountT));   // of this CTA
    int* digit_begin = digit_tot + padded;               // elements with a smaller digit
    int* digit_off = digit_begin + padded;               // ... and those with the digit in earlier CTAs
    // A segment of at most kInvBatch steps stays in registers: the count phase then also knows every
    // element's rank among the equal digits of its warp, so the scatter phase needs neither the
    // ballots nor the running counts again.
    const bool keep = seg <= 32 * kInvBatch;
    unsigned key[kInvBatch], val[kInvBatch];
    int local_rank[kInvBatch];

    // pass p reads (key, value) from src and writes to dst; pass 0 reads assign directly.  The position
    // in the last pass is final, and the member entries are written straight away.
    unsigned* key_buf[2] = {sort_a + 2 * ev_base, sort_b + 2 * ev_base};   // [E keys][E values] each
    for (int pass = 0; pass < n_pass; ++pass) {
        const int shift = pass * dbits;
        const bool last = pass == n_pass - 1;
        const unsigned* src_k = pass ? key_buf[(pass - 1) & 1] : nullptr;
        const unsigned* src_v = pass ? key_buf[(pass - 1) & 1] + E : nullptr;
        unsigned* dst_k = key_buf[pass & 1];
        unsigned* dst_v = key_buf[pass & 1] + E;
        auto load = [&](int b0) {                        // loads of kInvBatch steps together
#pragma unroll
            for (int q = 0; q < kInvBatch; ++q) {
                const int i = b0 + q * 32 + lane;
                key[q] = 0u;
                val[q] = (unsigned)i;
                if (i < s_end) {
                    if (pass) { key[q] = __ldcg(src_k + i); val[q] = __ldcg(src_v + i); }
                    else key[q] = (unsigned)assign[ev_base + i];
                }
            }
            if (pass) return;
#pragma unroll
            for (int q = 0; q < kInvBatch; ++q) {
                if (key[q] < (unsigned)B) continue;
                atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX);
                key[q] = 0u;
            }
        };
        // rank among the elements of the warp's segment with the same digit, which it counts
        auto rank_in_warp = [&](unsigned d, bool valid) {
            const unsigned peers = same_digit_lanes<kMaxBits>(d, valid, dbits);
            const int r = valid ? (int)cnt[warp * nd + d] + __popc(peers & lt_mask) : 0;
            __syncwarp();
            if (valid && (peers & lt_mask) == 0u) cnt[warp * nd + d] += (CountT)__popc(peers);
            __syncwarp();
            return r;
        };
        if (keep) load(s_begin);
        for (int i = threadIdx.x; i < (int)(kInvWarps * sizeof(CountT)) * padded / 16; i += kInvThreads)
            reinterpret_cast<uint4*>(cnt)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        for (int b0 = s_begin; b0 < s_end; b0 += 32 * kInvBatch) {
            if (!keep) load(b0);
#pragma unroll
            for (int q = 0; q < kInvBatch; ++q)
                if (b0 + q * 32 < s_end) local_rank[q] = rank_in_warp((key[q] >> shift) & dmask, b0 + q * 32 + lane < s_end);
        }
        __syncthreads();
        // exclusive scan over (digit major, warp minor): first over the warps, one 32-bit word of counts
        // at a time (two 16-bit sums stay apart) ...
        {
            constexpr int kPer = 4 / (int)sizeof(CountT);
            const int words = nd / kPer;
            unsigned* cw = reinterpret_cast<unsigned*>(cnt);
            for (int i = threadIdx.x; i < words; i += kInvThreads) {
                unsigned c[kInvWarps], tot = 0u;
#pragma unroll
                for (int w = 0; w < kInvWarps; ++w) c[w] = cw[w * words + i];
#pragma unroll
                for (int w = 0; w < kInvWarps; ++w) { cw[w * words + i] = tot; tot += c[w]; }
                if (kPer == 2) {
                    digit_tot[2 * i] = (int)(tot & 0xffffu);
                    digit_tot[2 * i + 1] = (int)(tot >> 16);
                } else {
                    digit_tot[i] = (int)tot;
                }
            }
            for (int i = nd + threadIdx.x; i < padded; i += kInvThreads) digit_tot[i] = 0;
        }
        sync();
        // ... then over the digit totals of all CTAs, four digits per thread
        {
            const int d0 = 4 * threadIdx.x;
            const bool mine = d0 < padded;
            int4 all = make_int4(0, 0, 0, 0), before = make_int4(0, 0, 0, 0);
            if (mine) {
#pragma unroll
                for (int c = 0; c < kInvMaxCluster; ++c) {
                    if (c >= ctas) continue;
                    const int4 x = ctas == 1 ? *reinterpret_cast<const int4*>(digit_tot + d0) : ptx::ld_cluster_int4(digit_tot + d0, c);
                    all.x += x.x; all.y += x.y; all.z += x.z; all.w += x.w;
                    if (c < cta) { before.x += x.x; before.y += x.y; before.z += x.z; before.w += x.w; }
                }
            }
            const int sum = all.x + all.y + all.z + all.w;
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            if (lane == 31) warp_sums[warp] = incl;
            __syncthreads();
            int base = incl - sum;
            for (int w = 0; w < warp; ++w) base += warp_sums[w];
            if (mine) {
                const int4 b = make_int4(base, base + all.x, base + all.x + all.y, base + all.x + all.y + all.z);
                *reinterpret_cast<int4*>(digit_begin + d0) = b;
                *reinterpret_cast<int4*>(digit_off + d0) = make_int4(b.x + before.x, b.y + before.y, b.z + before.z, b.w + before.w);
            }
        }
        __syncthreads();
        // scatter; the running counts of a segment that was not kept in registers go on from the scan's
        for (int b0 = s_begin; b0 < s_end; b0 += 32 * kInvBatch) {
            if (!keep) load(b0);
            int pe[kInvBatch];
            float w[kInvBatch];
#pragma unroll
            for (int q = 0; q < kInvBatch; ++q) {
                pe[q] = 0;
                w[q] = 1.0f;
                if (!last || b0 + q * 32 + lane >= s_end) continue;
                pe[q] = evict_idx[ev_base + val[q]];
                if (weighted) w[q] = sim[ev_base + val[q]];
            }
#pragma unroll
            for (int q = 0; q < kInvBatch; ++q) {
                if (b0 + q * 32 >= s_end) continue;
                const bool valid = b0 + q * 32 + lane < s_end;
                const unsigned d = (key[q] >> shift) & dmask;
                const int off = digit_off[d] + (keep ? (int)cnt[warp * nd + d] + local_rank[q] : rank_in_warp(d, valid));
                if (!valid) continue;
                if (last) {
                    if (pe[q] < 0 || pe[q] >= rq.L) { atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pe[q] = 0; }
                    ent[off + (int)key[q] + 1] = make_int2(pe[q], __float_as_int(w[q]));   // sits after key + 1 kept rows
                    if (pass) __stcg(dst_k + off, key[q]);
                } else {
                    __stcg(dst_k + off, key[q]);
                    __stcg(dst_v + off, val[q]);
                }
            }
        }
        sync();
    }
    if (n_pass == 1) {
        // digit = slot: digit_begin[c] is the first sorted index whose slot is >= c
        auto begin = [&](int c) { return c < nd ? digit_begin[c] : E; };
        for (int c = thread; c < B; c += n_threads) kept.write(c, kept_idx_head[c], begin(c), begin(c + 1) - begin(c));
        return;
    }
    // row boundaries: rp[c] = first sorted index whose slot is >= c
    const unsigned* fin_k = key_buf[(n_pass - 1) & 1];
    for (int i0 = thread; i0 < E; i0 += n_threads * kInvBatch) {
        int cur[kInvBatch], prev[kInvBatch];
#pragma unroll
        for (int q = 0; q < kInvBatch; ++q) {
            const int i = i0 + q * n_threads;
            cur[q] = i < E ? (int)__ldcg(fin_k + i) : 0;
            prev[q] = i < E && i ? (int)__ldcg(fin_k + i - 1) : -1;
        }
#pragma unroll
        for (int q = 0; q < kInvBatch; ++q) {
            const int i = i0 + q * n_threads;
            if (i >= E) continue;
            for (int c = prev[q] + 1; c <= cur[q]; ++c) __stcg(rp + c, i);
            if (i == E - 1) for (int c = cur[q] + 1; c <= B; ++c) __stcg(rp + c, E);
        }
    }
    sync();
    for (int c = thread; c < B; c += n_threads) {
        const int begin = __ldcg(rp + c);
        kept.write(c, kept_idx_head[c], begin, __ldcg(rp + c + 1) - begin);
    }
}

// The same result in one pass, a digit being a whole slot: every warp has a count per slot, in a byte, so
// that the sixteen counts of a slot are one 16-byte word and the sum over the warps before one's own four
// byte-wise dot products.  A warp's segment is at most kCountSeg elements and stays in registers.
// Every CTA of the cluster owns a share of the slots: it adds up the CTAs' totals of these, leaves each
// CTA the position of its first member per slot, and writes the kept rows' entries.  26214 evicted tokens
// x 8 heads into 6554 slots 42 us with two sorting passes, 25 counted; 13107 x 40 into 3277 46 and 32; 6554
// x 32 into 1638 (one sorting pass) 23.5 and 21.4; 7388 x 8 into 389 16.4 both.
constexpr int kCountSteps = kCountSeg / 32;
static_assert(kCountSeg % 32 == 0 && kCountSeg < 256 && kCountWarps == kInvWarps && kInvWarps == 16, "byte counts of sixteen warps");
constexpr int kCountBits = 13;
static_assert((1 << kCountBits) == kCountMaxSlots, "ballots per slot");
__device__ __forceinline__ int bytes_sum(const uint4& v, const uint4& m) {
    return (int)__dp4a(v.x, m.x, __dp4a(v.y, m.y, __dp4a(v.z, m.z, __dp4a(v.w, m.w, 0u))));
}

__global__ void __launch_bounds__(kInvThreads, 2)
invert_counting_kernel(const int* __restrict__ assign, const int* __restrict__ kept_idx, const int* __restrict__ evict_idx,
                       const float* __restrict__ sim, const __grid_constant__ ReqTable reqs, int n_kv_heads, int ctas, int max_slots,
                       long long T, int2* __restrict__ entries,
                       int4* __restrict__ unit_first, int* __restrict__ slot_cnt, int* status) {
    extern __shared__ __align__(16) unsigned char inv_smem[];
    __shared__ int warp_sums[kInvWarps];
    __shared__ int owner_tot[kInvMaxCluster];            // of this CTA's elements, those in each CTA's slots
    __shared__ int slots_begin;                          // elements in the slots of earlier CTAs
    uint4* cnt = reinterpret_cast<uint4*>(inv_smem);                                  // [slot] 16 warps
    int* off = reinterpret_cast<int*>(inv_smem + (size_t)max_slots * 16);             // [slot]
    unsigned short* tot = reinterpret_cast<unsigned short*>(off + max_slots);         // [slot]
    grid_dependency_wait();
    const Req rq = reqs.get(blockIdx.y);
    if (rq.mode == LOOKM_MERGE_NONE) return;             // its kept rows are copied, nothing is merged
    const int h = blockIdx.x / ctas, cta = blockIdx.x % ctas;     // the cluster: the CTAs of one head
    const int E = rq.E, B = rq.B;
    const long long ev_base = rq.ev_off + (long long)h * E;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    auto sync = [&]() { if (ctas > 1) ptx::cluster_sync(); else __syncthreads(); };
    int2* ent = entries + (long long)h * T + rq.tok_begin;
    const KeptEntries kept = {ent, unit_first + rq.unit_begin, slot_cnt + rq.kept_off + (long long)h * B, status,
                              rq.L, rq.unit_entries, h, n_kv_heads};
    const int* kept_idx_head = kept_idx + rq.kept_off + (long long)h * B;

    // the warp's elements
    const int seg = (E + ctas * kInvThreads - 1) / (ctas * kInvThreads) * 32;
    const int s_begin = min(E, (cta * kInvWarps + warp) * seg), s_end = min(E, s_begin + seg);
    unsigned key[kCountSteps];
    int pos[kCountSteps], local_rank[kCountSteps];
    float w[kCountSteps];
#pragma unroll
    for (int q = 0; q < kCountSteps; ++q) {
        const int i = s_begin + q * 32 + lane;
        key[q] = 0u;
        pos[q] = 0;
        w[q] = 1.0f;
        if (i >= s_end) continue;
        key[q] = (unsigned)assign[ev_base + i];
        pos[q] = evict_idx[ev_base + i];
        if (rq.mode == LOOKM_MERGE_WEIGHTED) w[q] = sim[ev_base + i];
    }
    for (int c = threadIdx.x; c < B; c += kInvThreads) cnt[c] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < kInvMaxCluster) owner_tot[threadIdx.x] = 0;
    if (threadIdx.x == 0) slots_begin = 0;
    int bits = 0;
    while ((1 << bits) < B) ++bits;
#pragma unroll
    for (int q = 0; q < kCountSteps; ++q) {
        if (key[q] >= (unsigned)B || pos[q] < 0 || pos[q] >= rq.L) {
            atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX);
            if (key[q] >= (unsigned)B) key[q] = 0u;
            if (pos[q] < 0 || pos[q] >= rq.L) pos[q] = 0;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kCountSteps; ++q) {
        if (s_begin + q * 32 >= s_end) continue;
        const bool valid = s_begin + q * 32 + lane < s_end;
        const unsigned peers = same_digit_lanes<kCountBits>(key[q], valid, bits);
        unsigned char* n = reinterpret_cast<unsigned char*>(cnt + key[q]) + warp;
        local_rank[q] = valid ? (int)*n + __popc(peers & lt_mask) : 0;
        __syncwarp();
        if (valid && (peers & lt_mask) == 0u) *n = (unsigned char)(*n + __popc(peers));
        __syncwarp();
    }
    __syncthreads();

    // this CTA's total of every slot, and of every CTA's share of the slots
    const int share = ((B + ctas - 1) / ctas + 3) / 4 * 4;         // (ctas * share <= max_slots)
    const uint4 ones = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
#pragma unroll
    for (int o = 0; o < kInvMaxCluster; ++o) {
        if (o >= ctas) continue;
        int sum = 0;
        for (int c = o * share + threadIdx.x; c < (o + 1) * share; c += kInvThreads) {
            const int t = c < B ? bytes_sum(cnt[c], ones) : 0;
            tot[c] = (unsigned short)t;
            sum += t;
        }
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0 && sum) atomicAdd(&owner_tot[o], sum);
    }
    sync();
    if (threadIdx.x < kInvMaxCluster * kInvMaxCluster) {
        const int c = threadIdx.x / kInvMaxCluster, o = threadIdx.x % kInvMaxCluster;
        if (c < ctas && o < cta) atomicAdd(&slots_begin, ptx::ld_cluster_int(&owner_tot[o], c));
    }
    // own slots, four per thread: members before each, and where every CTA's first one goes
    for (int t0 = 0, run = 0; t0 < share; t0 += 4 * kInvThreads) {
        const int d0 = cta * share + t0 + 4 * threadIdx.x;
        const bool mine = t0 + 4 * threadIdx.x < share;
        uint2 x[kInvMaxCluster];
        int pc[4] = {0, 0, 0, 0}, all[4] = {0, 0, 0, 0};
#pragma unroll
        for (int c = 0; c < kInvMaxCluster; ++c) {
            x[c] = make_uint2(0u, 0u);
            if (mine && c < ctas)
                x[c] = ctas > 1 ? ptx::ld_cluster_uint2(tot + d0, c) : *reinterpret_cast<const uint2*>(tot + d0);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (mine && d0 + j < B) pc[j] = kept_idx_head[d0 + j];
#pragma unroll
        for (int c = 0; c < kInvMaxCluster; ++c) {
            all[0] += x[c].x & 0xffffu;
            all[1] += x[c].x >> 16;
            all[2] += x[c].y & 0xffffu;
            all[3] += x[c].y >> 16;
        }
        const int sum = all[0] + all[1] + all[2] + all[3];
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();                                 // slots_begin; the last turn's warp_sums have been read
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        int begin = slots_begin + run + incl - sum;
        for (int v = 0; v < kInvWarps; ++v) {
            if (v < warp) begin += warp_sums[v];
            run += warp_sums[v];
        }
        if (!mine) continue;
        int4 at = make_int4(begin, begin + all[0], begin + all[0] + all[1], begin + all[0] + all[1] + all[2]);
        const int first[4] = {at.x, at.y, at.z, at.w};
#pragma unroll
        for (int c = 0; c < kInvMaxCluster; ++c) {
            if (c >= ctas) continue;
            if (ctas > 1) ptx::st_cluster_int4(off + d0, c, at);
            else *reinterpret_cast<int4*>(off + d0) = at;
            at.x += x[c].x & 0xffffu;
            at.y += x[c].x >> 16;
            at.z += x[c].y & 0xffffu;
            at.w += x[c].y >> 16;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (d0 + j < B) kept.write(d0 + j, pc[j], first[j], all[j]);
        }
    }
    sync();

    const auto before = [&](int v) {                     // ones in the bytes of word v that belong to earlier warps
        const int n = min(max(warp - 4 * v, 0), 4);
        return n == 4 ? 0x01010101u : 0x01010101u & ((1u << (8 * n)) - 1u);
    };
    const uint4 earlier = make_uint4(before(0), before(1), before(2), before(3));
#pragma unroll
    for (int q = 0; q < kCountSteps; ++q) {
        if (s_begin + q * 32 + lane >= s_end) continue;
        // sits after key + 1 kept rows
        const int at = off[key[q]] + bytes_sum(cnt[key[q]], earlier) + local_rank[q] + (int)key[q] + 1;
        ent[at] = make_int2(pos[q], __float_as_int(w[q]));
    }
}

// ---------------------------------------------------------------------------------------------
// Merge + compact (Eq. 6-7, 10-12).  Every K and V row of the prompt is read exactly once: the
// entry list of a (request, head) names, slot by slot, the kept row and then its members.  A warp
// takes a work unit of unit_entries consecutive entries (sized so that each warp gets about one
// unit, at least 32 entries), fetches the rows 8 entries at a time with 16-byte cp.async copies
// into its own shared-memory ring (three buffers; every lane later reads back exactly the bytes it
// copied, so cp.async.wait_group is all the synchronisation needed), and walks the staged rows in
// order: lanes 0-15 hold the K row, lanes 16-31 the V row, 16 bytes per lane, fp32 accumulation in
// member order, one rounding.
//   averaged : (x_c + sum x_e) / (n + 1)                       (Eq. 10)
//   pivotal  : (x_c + 1/2 sum (x_e + x_c)) / (n + 1)           (Eq. 11)
//   weighted : (x_c + sum sim_e x_e) / (n + 1)                 (Eq. 12)
// A row without members is copied bit for bit.
//
// Units are cut at fixed entry counts, not at slot boundaries, so that every warp has the same
// amount to read however skewed the member counts are.  A slot whose entries straddle units is
// summed piecewise: every unit that holds a piece stores its fp32 partial sum (the unit with the
// kept row also stores that row) in its own record, then bumps the slot's arrival counter; the
// warp that arrives last adds the pieces in unit order and writes the row.  Nobody waits for
// anybody, and the order of the additions does not depend on who came last.
// ---------------------------------------------------------------------------------------------
constexpr int kMergeWarps = 16;                      // per CTA; one CTA per SM
constexpr int kChunk = 8;                            // entries staged per buffer
constexpr int kRing = 3;                             // buffers per warp: two chunks in flight while one is read
constexpr int kRowBytes = kHeadDim * 2;              // one bf16 row of K or V
// Record of a unit: [0, 1024) partial sums of its leading piece (slot begun in an earlier unit),
// [1024, 2048) partial sums of its trailing piece (slot that goes on in the next unit),
// [2048, 2560) the kept K|V row of the trailing piece.  Per piece: 8 floats (or 16 bytes) per lane.
constexpr int kPartFloats = kMergePartBytes / 4;

struct MergeShared {
    alignas(128) uint8_t rows[kMergeWarps][kRing][kChunk][2 * kRowBytes];   // [warp][buffer][entry][K|V]
};

// (only: reqs.only in shared memory)
__device__ __forceinline__ const Req& find_req_by_unit(const ReqTable& reqs, const Req& only, long long g) {
    if (reqs.n == 1) return only;
    int lo = 0, hi = reqs.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long long)reqs.rows[mid].unit_begin <= g) lo = mid; else hi = mid - 1;
    }
    return reqs.rows[lo];
}

__device__ __forceinline__ float4 ld_cg_f4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }

__global__ void __launch_bounds__(kMergeWarps * 32)
merge_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
             long long stride_tok, long long stride_head, const __grid_constant__ ReqTable reqs,
             int n_kv_heads, long long T, long long total_units, const int2* __restrict__ entries,
             const int4* __restrict__ unit_first, int* __restrict__ slot_cnt, float* __restrict__ parts,
             int varlen_output, long long out_stride_head, __nv_bfloat16* __restrict__ out_k,
             __nv_bfloat16* __restrict__ out_v) {
    extern __shared__ uint8_t merge_smem_raw[];
    MergeShared& sh = *reinterpret_cast<MergeShared*>(
        (reinterpret_cast<uintptr_t>(merge_smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l16 = lane & 15;
    const uint32_t buf0 = (uint32_t)__cvta_generic_to_shared(&sh.rows[warp][0][0][0]) + lane * 16;
    const __nv_bfloat16* tensor = lane < 16 ? k : v;
    __nv_bfloat16* dst_base = lane < 16 ? out_k : out_v;
    const unsigned tok_bytes = (unsigned)stride_tok * 2u;      // the launcher checks that this fits
    uint32_t n_chunks_done = 0;                      // chunks this warp has consumed (buffer parity)
    __shared__ Req only;
    if (reqs.n == 1) copy_words(only, reqs.only);
    __syncthreads();
    grid_dependency_wait();

    for (long long g = (long long)blockIdx.x * kMergeWarps + warp; g < total_units;
         g += (long long)gridDim.x * kMergeWarps) {
        const Req& rq = find_req_by_unit(reqs, only, g);
        const int L = rq.L, B = rq.B, mode = rq.mode, ue = rq.unit_entries;
        const long long ul = g - rq.unit_begin;
        // heads vary fastest: warps running at the same time then read the same token range of
        // different heads, i.e. neighbouring 256-byte rows of the same DRAM pages
        const int h = (int)(ul % n_kv_heads), u = (int)(ul / n_kv_heads);
        const int e_lo = u * ue, e_hi = min(L, e_lo + ue);
        int4 first = make_int4(0, 0, 0, 0);           // slot of the first entry; its first entry, member count
        if (lane == 0) first = __ldg(unit_first + g); // needed at the first kept row at the earliest
        int* cnt = slot_cnt + rq.kept_off + (long long)h * B;
        const int2* ent = entries + (long long)h * T + rq.tok_begin;
        const char* src = reinterpret_cast<const char*>(tensor + (long long)rq.tok_begin * stride_tok +
                                                        (long long)h * stride_head + l16 * 8);
        const int n_chunks = (e_hi - e_lo + kChunk - 1) / kChunk;

        // entry metadata of a chunk (lanes 0-7: one entry each)
        auto load_meta = [&](int kc, int& pos, float& w) {
            pos = 0;
            w = 0.f;
            const int e = e_lo + kc * kChunk + lane;
            if (lane < kChunk && kc < n_chunks && e < e_hi) { const int2 x = ent[e]; pos = x.x; w = __int_as_float(x.y); }
        };
        // start the row copies of chunk kc: for every entry, lanes 0-15 copy its K row and lanes
        // 16-31 its V row, 16 bytes each; one commit group per chunk
        auto issue = [&](int kc, int pos) {
            const int n_ent = min(kChunk, e_hi - e_lo - kc * kChunk);    // <= 0 past the unit: empty group
            const uint32_t dst = buf0 + ((n_chunks_done + (uint32_t)kc) % kRing) * (kChunk * 2 * kRowBytes);
#pragma unroll
            for (int q = 0; q < kChunk; ++q) {
                const unsigned tok = (unsigned)__shfl_sync(0xffffffffu, pos, q) & 0x7fffffffu;
                if (q < n_ent)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                 ::"r"(dst + q * (2 * kRowBytes)), "l"(src + (size_t)tok * tok_bytes)
                                 : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };

        int pos_a, pos_b, pos_c;
        float w_a, w_b, w_c;
        load_meta(0, pos_a, w_a);
        load_meta(1, pos_b, w_b);
        load_meta(2, pos_c, w_c);
        issue(0, pos_a);
        issue(1, pos_b);

        // running piece: the slot, whether its kept row was met in this unit (and at which entry),
        // the members met
        const bool starts_with_kept = __shfl_sync(0xffffffffu, pos_a, 0) < 0;
        const int first_slot = __shfl_sync(0xffffffffu, first.x, 0);
        int slot = starts_with_kept ? first_slot - 1 : first_slot;
        bool active = !starts_with_kept, have_kept = false;
        bool lead_piece = false, trail_piece = false;    // pieces of shared slots this unit has stored
        int n_mem = 0, n_seen = 0, kept_entry = 0;
        uint4 raw_c = make_uint4(0u, 0u, 0u, 0u);
        float acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.f;

        auto write_row = [&](int c, const uint4& kept_raw, const float* sum, int n) {
            uint4 result = kept_raw;
            if (n > 0) {
                const Row8 xc = unpack8(kept_raw);
                const float inv = 1.0f / (float)(n + 1);
                // pivotal: each member contributes (x_e + x_c) / 2
                const float wc = (mode == LOOKM_MERGE_PIVOTAL) ? 1.f + 0.5f * (float)n : 1.f;
                const float wm = (mode == LOOKM_MERGE_PIVOTAL) ? 0.5f : 1.f;
                Row8 o;
#pragma unroll
                for (int i = 0; i < 8; ++i) o.v[i] = fmaf(wc, xc.v[i], wm * sum[i]) * inv;
                result = pack8(o);
            }
            long long at;
            if (varlen_output) at = (((long long)rq.out_begin + c) * n_kv_heads + h) * kHeadDim;
            else at = (long long)h * out_stride_head + (long long)c * kHeadDim;
            *reinterpret_cast<uint4*>(dst_base + at + l16 * 8) = result;
        };
        // ends the running piece: a whole slot is written out; a piece of a slot that other units
        // share goes to this unit's record (announced after the loop)
        auto flush = [&]() {
            if (!active) return;
            if (have_kept && n_seen == n_mem) {
                write_row(slot, raw_c, acc, n_mem);
                return;
            }
            float* rec = parts + g * kPartFloats + (have_kept ? 256 : 0) + lane * 8;
            *reinterpret_cast<float4*>(rec) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            *reinterpret_cast<float4*>(rec + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
            if (have_kept) {
                *reinterpret_cast<uint4*>(parts + g * kPartFloats + 512 + lane * 4) = raw_c;
                trail_piece = true;
            } else {
                lead_piece = true;
            }
        };
        // adds the pieces of slot c (kept row in unit u0, last member in unit u1) in unit order
        auto combine = [&](int c, int u0, int u1, int n) {
            const float* r0 = parts + ((long long)rq.unit_begin + (long long)u0 * n_kv_heads + h) * kPartFloats;
            float sum[8];
            {
                const float4 lo = ld_cg_f4(r0 + 256 + lane * 8), hi = ld_cg_f4(r0 + 256 + lane * 8 + 4);
                sum[0] = lo.x; sum[1] = lo.y; sum[2] = lo.z; sum[3] = lo.w;
                sum[4] = hi.x; sum[5] = hi.y; sum[6] = hi.z; sum[7] = hi.w;
            }
            const uint4 kept_raw = __ldcg(reinterpret_cast<const uint4*>(r0 + 512 + lane * 4));
            for (int uu = u0 + 1; uu <= u1; ++uu) {
                const float* r = r0 + (long long)(uu - u0) * n_kv_heads * kPartFloats;
                const float4 lo = ld_cg_f4(r + lane * 8), hi = ld_cg_f4(r + lane * 8 + 4);
                sum[0] += lo.x; sum[1] += lo.y; sum[2] += lo.z; sum[3] += lo.w;
                sum[4] += hi.x; sum[5] += hi.y; sum[6] += hi.z; sum[7] += hi.w;
            }
            write_row(c, kept_raw, sum, n);
        };

        for (int kc = 0; kc < n_chunks; ++kc) {
            // chunk kc + 2 goes to the buffer whose rows were consumed one iteration ago; a commit
            // group is made for every chunk index (empty past the unit), so "all but the two
            // newest groups" always means: chunk kc has landed
            issue(kc + 2, pos_c);
            int pos_d;
            float w_d;
            load_meta(kc + 3, pos_d, w_d);
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            const int n_ent = min(kChunk, e_hi - e_lo - kc * kChunk);
            const uint32_t rows = buf0 + ((n_chunks_done + (uint32_t)kc) % kRing) * (kChunk * 2 * kRowBytes);
            uint4 x[kChunk];                         // this lane's 16 bytes of every staged row
#pragma unroll
            for (int q = 0; q < kChunk; ++q)
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(x[q].x), "=r"(x[q].y), "=r"(x[q].z), "=r"(x[q].w)
                             : "r"(rows + q * (2 * kRowBytes)));
#pragma unroll
            for (int q = 0; q < kChunk; ++q) {
                const int pe = __shfl_sync(0xffffffffu, pos_a, q);
                const float w = __shfl_sync(0xffffffffu, w_a, q);
                if (q >= n_ent) break;
                if (pe < 0) {                        // a kept row starts the next slot
                    flush();
                    ++slot;
                    active = true;
                    have_kept = true;
                    raw_c = x[q];
                    n_mem = (int)w;
                    n_seen = 0;
                    kept_entry = e_lo + kc * kChunk + q;
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
                } else {
                    const Row8 xe = unpack8(x[q]);
                    ++n_seen;
#pragma unroll
                    for (int i = 0; i < 8; ++i) acc[i] = fmaf(w, xe.v[i], acc[i]);
                }
            }
            __syncwarp();
            pos_a = pos_b; w_a = w_b;
            pos_b = pos_c; w_b = w_c;
            pos_c = pos_d; w_c = w_d;
        }
        flush();
        n_chunks_done += (uint32_t)n_chunks;
        if (lead_piece || trail_piece) {
            // announce the stored pieces (lane 0: the leading one, lane 1: the trailing one); the
            // unit that arrives last at a slot finishes its row
            __threadfence();
            __syncwarp();
            int c = 0, s0 = 0, n = 0;
            bool mine = false;
            if (lane == 0 && lead_piece) { c = first.x; s0 = first.y; n = first.z; mine = true; }
            if (lane == 1 && trail_piece) { c = slot; s0 = kept_entry; n = n_mem; mine = true; }
            const int u0 = s0 / ue, u1 = (s0 + n) / ue;          // units of the kept row / the last member
            const bool last = mine && atomicAdd(cnt + c, 1) == u1 - u0;
            const unsigned finish = __ballot_sync(0xffffffffu, last);
            if (finish) __threadfence();
            for (int which = 0; which < 2; ++which)
                if (finish & (1u << which))
                    combine(__shfl_sync(0xffffffffu, c, which), __shfl_sync(0xffffffffu, u0, which),
                            __shfl_sync(0xffffffffu, u1, which), __shfl_sync(0xffffffffu, n, which));
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Inversion, merge and compaction in one launch, for short prompts.  There the two kernels above are
// chains of round trips (table, lists, sort, entry list in memory, metadata, rows, records, counters) and a launch, not bandwidth.  A CTA owns the slots [c0, c1) of one (request, head): it
// sorts the evicted tokens of its slots by slot (stable, counters in shared memory), keeps the entry
// list in shared memory, and its warps walk equal shares of that list.  A slot whose entries straddle
// shares is summed piecewise through shared memory, pieces in share order.
// lookm_merge as a whole, two kernels | one (us, graph replay): 700 tokens x 32 heads 26.7 | 16.4,
// 2048 x 8 28.7 | 14.7, 2048 x 32 30.1 | 23.0, 4096 x 8 30.8 | 20.5, 4096 x 32 37.4 | 34.9; batches, where one CTA
// has a whole head: 200 prompts of 100 x 32 466 | 200, 16 of 1000 x 32 166 | 89, 64 of 1000 x 8 171 | 94, 16 of 4000
// x 32 364 | 334.  Every CTA of a head sorts the whole evicted list, so the gain is gone soon after
// kMergeShortMax.
// ---------------------------------------------------------------------------------------------
constexpr int kFuseThreads = 512;
constexpr int kFuseWarps = kFuseThreads / 32;
constexpr int kFuseBatch = 8;                        // rows requested together by a warp

struct FuseShared {
    float lead[kFuseWarps][32][8];                   // piece of a slot begun in an earlier share
    int warp_sums[kFuseWarps];
};
// dynamic shared memory behind it: counters u16 [warp][slot], offsets int [slot + 1], entries {pos, weight}
__host__ __device__ inline size_t fuse_smem(int max_slots, int max_L) {
    return sizeof(FuseShared) + (size_t)((kFuseWarps * max_slots * 2 + 15) / 16 * 16) + (size_t)((max_slots + 4) / 4 * 16) +
           (size_t)max_L * 8;
}

// kSteps: 32-token steps of a warp's segment of the evicted list (E <= 512 kSteps).
template <int kSteps>
__global__ void __launch_bounds__(kFuseThreads, 2)
merge_short_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v, long long stride_tok,
                   long long stride_head, const int* __restrict__ assign, const int* __restrict__ kept_idx,
                   const int* __restrict__ evict_idx, const float* __restrict__ sim, const Req* __restrict__ reqs,
                   int n_kv_heads, int max_slots, int varlen_output, long long out_stride_head,
                   __nv_bfloat16* __restrict__ out_k, __nv_bfloat16* __restrict__ out_v, int* status) {
    extern __shared__ __align__(16) unsigned char fuse_raw[];
    FuseShared& sh = *reinterpret_cast<FuseShared*>(fuse_raw);
    unsigned short* cnt = reinterpret_cast<unsigned short*>(fuse_raw + sizeof(FuseShared));
    int* first = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(cnt) + (kFuseWarps * max_slots * 2 + 15) / 16 * 16);
    int2* ent = reinterpret_cast<int2*>(reinterpret_cast<unsigned char*>(first) + (max_slots + 4) / 4 * 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    grid_dependency_wait();
    // From the table, also of a single prompt: the walk has no registers for a request from either of two places
    // (28.8 | 31.4 us for 2900 tokens x 40 heads, 109 | 130 us for five prompts of 1800 to 2800 x 32; by way of shared
    // memory 32.2 and 130).
    const Req rq = reqs[blockIdx.z];
    if (rq.mode == LOOKM_MERGE_NONE) return;
    const int h = blockIdx.y;
    const int E = rq.E, B = rq.B, mode = rq.mode;
    const int per = (B + (int)gridDim.x - 1) / (int)gridDim.x;       // slots per CTA, at most max_slots
    const int c0 = min(B, (int)blockIdx.x * per), n_slots = min(B, c0 + per) - c0;
    if (n_slots <= 0) return;
    const long long ev_base = rq.ev_off + (long long)h * E, kept_base = rq.kept_off + (long long)h * B;

    // ---- the evicted tokens' lists are requested at once (the kept positions when the entries are written) ----
    const int seg = ((E + kFuseWarps * 32 - 1) / (kFuseWarps * 32)) * 32;
    const int s_begin = warp * seg;
    int key[kSteps], pos[kSteps];
    float wgt[kSteps];
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
        const int i = s_begin + q * 32 + lane;
        key[q] = -1;
        pos[q] = 0;
        wgt[q] = 1.f;
        if (q * 32 < seg && i < E) {
            key[q] = assign[ev_base + i];
            pos[q] = evict_idx[ev_base + i];
            if (mode == LOOKM_MERGE_WEIGHTED) wgt[q] = sim[ev_base + i];
        }
    }
    for (int i = threadIdx.x; i < kFuseWarps * n_slots; i += kFuseThreads) cnt[i] = 0;
    __syncthreads();
    // ---- rank of every token among its warp's tokens of the same slot ----
    int dbits = 1;
    while ((1 << dbits) < n_slots) ++dbits;
    unsigned short* my_cnt = cnt + warp * n_slots;
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
        if (q * 32 >= seg) break;
        const int i = s_begin + q * 32 + lane;
        if (i < E && (unsigned)key[q] >= (unsigned)B) { atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); key[q] = 0; }
        const int d = key[q] - c0;
        const bool valid = i < E && (unsigned)d < (unsigned)n_slots;
        key[q] = -1;
        const unsigned any = __ballot_sync(0xffffffffu, valid);
        if (any == 0u) continue;
        unsigned peers = any;
        for (int b = 0; b < dbits; ++b) {
            const bool bit = (d >> b) & 1;
            const unsigned bal = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bal : ~bal;
        }
        if (valid) key[q] = (d << 16) | ((int)my_cnt[d] + __popc(peers & lt_mask));
        __syncwarp();
        if (valid && (peers & lt_mask) == 0u) my_cnt[d] += (unsigned short)__popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // ---- members per slot, then the slots' places in the entry list (kept row + members each) ----
    int run = 0;
    for (int d0 = 0; d0 < n_slots; d0 += kFuseThreads) {
        const int d = d0 + threadIdx.x;
        int tot = 0;
        if (d < n_slots) {
#pragma unroll
            for (int w = 0; w < kFuseWarps; ++w) {
                const int c = cnt[w * n_slots + d];
                cnt[w * n_slots + d] = (unsigned short)tot;
                tot += c;
            }
            ++tot;                                   // the kept row
        }
        int incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        if (lane == 31) sh.warp_sums[warp] = incl;
        __syncthreads();
        int before = run, all = run;
#pragma unroll
        for (int w = 0; w < kFuseWarps; ++w) {
            const int x = sh.warp_sums[w];
            before += w < warp ? x : 0;
            all += x;
        }
        if (d < n_slots) first[d] = before + incl - tot;
        run = all;
        __syncthreads();
    }
    const int n_ent = run;
    if (threadIdx.x == 0) first[n_slots] = n_ent;
    __syncthreads();
    for (int c = threadIdx.x; c < n_slots; c += kFuseThreads) {
        int pc = kept_idx[kept_base + c0 + c];
        if (pc < 0 || pc >= rq.L) { atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pc = 0; }
        ent[first[c]] = make_int2(pc | (int)0x80000000, c);
    }
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
        if (key[q] < 0) continue;
        const int d = key[q] >> 16;
        if (pos[q] < 0 || pos[q] >= rq.L) { atomicExch(status, (int)LOOKM_ERR_DEVICE_BAD_INDEX); pos[q] = 0; }
        ent[first[d] + 1 + (int)my_cnt[d] + (key[q] & 0xffff)] = make_int2(pos[q], __float_as_int(wgt[q]));
    }
    __syncthreads();

    // ---- walk: lanes 0-15 hold the K row, 16-31 the V row, 16 bytes per lane ----
    const int l16 = lane & 15;
    const __nv_bfloat16* src = (lane < 16 ? k : v) + (long long)rq.tok_begin * stride_tok + (long long)h * stride_head + l16 * 8;
    __nv_bfloat16* dst = (lane < 16 ? out_k : out_v) + l16 * 8;
    auto write_row = [&](int d, const uint4& kept_raw, const float (&sum)[8], int n) {
        uint4 result = kept_raw;
        if (n > 0) {
            const Row8 xc = unpack8(kept_raw);
            const float inv = 1.0f / (float)(n + 1);
            const float wc = (mode == LOOKM_MERGE_PIVOTAL) ? 1.f + 0.5f * (float)n : 1.f;
            const float wm = (mode == LOOKM_MERGE_PIVOTAL) ? 0.5f : 1.f;
            Row8 o;
#pragma unroll
            for (int i = 0; i < 8; ++i) o.v[i] = fmaf(wc, xc.v[i], wm * sum[i]) * inv;
            result = pack8(o);
        }
        const int c = c0 + d;
        long long at;
        if (varlen_output) at = (((long long)rq.out_begin + c) * n_kv_heads + h) * kHeadDim;
        else at = (long long)h * out_stride_head + (long long)c * kHeadDim;
        *reinterpret_cast<uint4*>(dst + at) = result;
    };
    const int share = max(kFuseBatch, (n_ent + kFuseWarps - 1) / kFuseWarps);
    const int e_lo = min(n_ent, warp * share), e_hi = min(n_ent, e_lo + share);
    float acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    uint4 raw_c = make_uint4(0u, 0u, 0u, 0u);
    int d = -1;                                      // running slot; -1: begun in an earlier share
    const bool open = e_lo < e_hi && ent[e_lo].x >= 0;       // the share starts inside a slot
    auto flush = [&]() {                             // the running slot is complete, or was begun elsewhere
        if (d >= 0) {
            write_row(d, raw_c, acc, first[d + 1] - first[d] - 1);
        } else if (open) {
#pragma unroll
            for (int i = 0; i < 8; ++i) sh.lead[warp][lane][i] = acc[i];
        }
    };
    for (int e0 = e_lo; e0 < e_hi; e0 += kFuseBatch) {
        int2 en[kFuseBatch];
        uint4 x[kFuseBatch];
#pragma unroll
        for (int q = 0; q < kFuseBatch; ++q) {
            en[q] = e0 + q < e_hi ? ent[e0 + q] : make_int2(0, 0);
            if (e0 + q < e_hi)
                x[q] = __ldg(reinterpret_cast<const uint4*>(src + (long long)(en[q].x & 0x7fffffff) * stride_tok));
        }
#pragma unroll
        for (int q = 0; q < kFuseBatch; ++q) {
            if (e0 + q >= e_hi) break;
            if (en[q].x < 0) {                       // a kept row starts the next slot
                flush();
                d = en[q].y;
                raw_c = x[q];
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = 0.f;
            } else {
                const Row8 xe = unpack8(x[q]);
                const float w = __int_as_float(en[q].y);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = fmaf(w, xe.v[i], acc[i]);
            }
        }
    }
    const bool goes_on = d >= 0 && first[d + 1] > e_hi;
    if (!goes_on && e_lo < e_hi) flush();
    __syncthreads();
    if (goes_on) {                                   // the share that has the kept row adds the pieces
        const int w1 = (first[d + 1] - 1) / share;   // share of the slot's last entry
        for (int w = warp + 1; w <= w1; ++w)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += sh.lead[w][lane][i];
        write_row(d, raw_c, acc, first[d + 1] - first[d] - 1);
    }
}

__global__ void __launch_bounds__(256)
write_table_kernel(const __grid_constant__ ReqChunk chunk, int count, Req* dst, int* clear, size_t n_clear) {
    grid_dependency_wait();
    const int i = threadIdx.x;
    if (blockIdx.x == 0 && i < count) dst[i] = chunk.r[i];
    for (size_t j = (size_t)blockIdx.x * blockDim.x + i; j < n_clear; j += (size_t)gridDim.x * blockDim.x) clear[j] = 0;
}

}  // namespace

cudaError_t launch_write_table(const ReqChunk& chunk, int count, Req* dst, int* clear, size_t n_clear, cudaStream_t stream) {
    const size_t blocks = n_clear / 2048 + 1;            // eight words per thread
    return launch_chained(write_table_kernel, dim3((unsigned)(blocks < 148 ? blocks : 148)), dim3(256), 0, stream, chunk, count,
                          dst, clear, n_clear);
}

cudaError_t launch_key_norms(const void* k, long long stride_tok, long long stride_head,
                             int n_kv_heads, long long T, float* rnorm_all, cudaStream_t stream) {
    const long long rows = T * n_kv_heads;
    if (rows <= 0) return cudaSuccess;
    long long blocks = (rows + 15) / 16;
    if (blocks > 148 * 32) blocks = 148 * 32;
    key_norms_kernel<<<(int)blocks, 256, 0, stream>>>((const __nv_bfloat16*)k, stride_tok, stride_head,
                                                      n_kv_heads, T, rnorm_all);
    return cudaGetLastError();
}

cudaError_t launch_gather_kept(const void* k, long long stride_tok, long long stride_head,
                               const ReqTable& reqs, int n_kv_heads, long long T,
                               long long total_kept_rows, const int* kept_idx,
                               const float* rnorm_all, void* kept_keys, float* rnorm_kept,
                               int* status, cudaStream_t stream) {
    if (total_kept_rows <= 0) return cudaSuccess;
    const long long blocks = (total_kept_rows + 15) / 16;
    return launch_chained(gather_kept_kernel, dim3((unsigned)blocks), dim3(256), 0, stream,
                          (const __nv_bfloat16*)k, stride_tok, stride_head, reqs, n_kv_heads, T,
                          total_kept_rows, kept_idx, rnorm_all, (__nv_bfloat16*)kept_keys, rnorm_kept,
                          status);
}

cudaError_t launch_invert_assignment(const int* assign, const int* kept_idx, const int* evict_idx,
                                     const float* sim, const ReqTable& reqs, int n_kv_heads, int ctas,
                                     long long T, bool wide_counts, int digit_bits, int* row_begin,
                                     int2* entries, int4* unit_first, int* slot_cnt,
                                     unsigned* sort_a, unsigned* sort_b, int* status,
                                     cudaStream_t stream) {
    // counters of the widest digit any request of the call needs: per warp, and three totals
    const auto bytes = [](int count, int bits) { return (size_t)(kInvWarps * count + 3 * (int)sizeof(int)) << (bits < 2 ? 2 : bits); };
    auto* narrow = invert_assignment_kernel<unsigned short, kInvDigitBits16>;
    auto* wide = invert_assignment_kernel<unsigned, kInvDigitBits32>;
    // the shared-memory limit is raised once per device to the most either instantiation can ask for
    static unsigned long long configured = 0;
    cudaError_t err = once_per_device(configured, [&]() {
        cudaError_t e = cudaFuncSetAttribute(narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(2, kInvDigitBits16));
        return e != cudaSuccess ? e : cudaFuncSetAttribute(wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(4, kInvDigitBits32));
    });
    if (err != cudaSuccess) return err;
    return launch_chained_clusters(wide_counts ? wide : narrow, dim3((unsigned)(n_kv_heads * ctas), (unsigned)reqs.n), dim3(kInvThreads),
                                   (unsigned)ctas, bytes(wide_counts ? 4 : 2, digit_bits), stream, assign, kept_idx, evict_idx, sim,
                                   reqs, n_kv_heads, ctas, T, row_begin, entries, unit_first, slot_cnt, sort_a, sort_b, status);
}

cudaError_t launch_invert_counting(const int* assign, const int* kept_idx, const int* evict_idx, const float* sim, const ReqTable& reqs,
                                   int n_kv_heads, int ctas, int max_slots, long long T, int2* entries,
                                   int4* unit_first, int* slot_cnt, int* status, cudaStream_t stream) {
    static unsigned long long configured = 0;
    cudaError_t err = once_per_device(configured, [&]() {
        return cudaFuncSetAttribute(invert_counting_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (kCountMaxSlots + 4 * kInvMaxCluster) * kCountSlotBytes);
    });
    if (err != cudaSuccess) return err;
    return launch_chained_clusters(invert_counting_kernel, dim3((unsigned)(n_kv_heads * ctas), (unsigned)reqs.n), dim3(kInvThreads),
                                   (unsigned)ctas, (size_t)max_slots * kCountSlotBytes, stream, assign, kept_idx, evict_idx, sim,
                                   reqs, n_kv_heads, ctas, max_slots, T, entries, unit_first, slot_cnt, status);
}

int merge_warps_per_sm() { return kMergeWarps; }

cudaError_t launch_merge(const void* k, const void* v, long long stride_tok, long long stride_head,
                         const ReqTable& reqs, int n_kv_heads, long long T,
                         long long total_units, const int2* entries,
                         const int4* unit_first, int* slot_cnt, float* parts,
                         int varlen_output, long long out_stride_head, void* out_k, void* out_v,
                         int num_sms, cudaStream_t stream) {
    if (total_units <= 0) return cudaSuccess;
    if (stride_tok <= 0 || stride_tok >= (1ll << 31)) return cudaErrorInvalidValue;   // byte stride kept in 32 bits
    const int smem = (int)sizeof(MergeShared) + 128;
    static unsigned long long configured = 0;
    cudaError_t err = once_per_device(configured, [&]() {
        return cudaFuncSetAttribute(merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    });
    if (err != cudaSuccess) return err;
    long long blocks = (total_units + kMergeWarps - 1) / kMergeWarps;
    if (blocks > num_sms) blocks = num_sms;              // persistent: one CTA per SM
    return launch_chained(merge_kernel, dim3((unsigned)blocks), dim3(kMergeWarps * 32), (size_t)smem, stream,
                          (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, stride_tok, stride_head, reqs,
                          n_kv_heads, T, total_units, entries, unit_first, slot_cnt,
                          parts, varlen_output, out_stride_head, (__nv_bfloat16*)out_k, (__nv_bfloat16*)out_v);
}

// Parts per (request, head): about two CTAs per SM, at least eight slots each.
cudaError_t launch_merge_short(const void* k, const void* v, long long stride_tok, long long stride_head, const int* assign,
                               const int* kept_idx, const int* evict_idx, const float* sim, const ReqTable& reqs,
                               int n_kv_heads, int max_L, int max_E, int max_B, int varlen_output, long long out_stride_head,
                               void* out_k, void* out_v, int* status, int num_sms, cudaStream_t stream) {
    const long long heads = (long long)n_kv_heads * reqs.n;
    long long parts = 2ll * num_sms / heads;             // one wave: two CTAs fit on an SM
    if (parts < 1) parts = 1;
    if (parts > (max_B + 7) / 8) parts = (max_B + 7) / 8;
    const int max_slots = (max_B + (int)parts - 1) / (int)parts;
    const size_t smem = fuse_smem(max_slots, max_L);
    static unsigned long long configured = 0;
    cudaError_t err = once_per_device(configured, [&]() {
        const int most = (int)fuse_smem(kMergeShortMax, kMergeShortMax);
        cudaError_t e = cudaFuncSetAttribute(merge_short_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(merge_short_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        return e;
    });
    if (err != cudaSuccess) return err;
    auto kernel = max_E <= 2 * kFuseThreads ? merge_short_kernel<2> : merge_short_kernel<8>;
    return launch_chained(kernel, dim3((unsigned)parts, (unsigned)n_kv_heads, (unsigned)reqs.n), dim3(kFuseThreads), smem, stream,
                          (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, stride_tok, stride_head, assign, kept_idx, evict_idx,
                          sim, reqs.rows, n_kv_heads, max_slots, varlen_output, out_stride_head, (__nv_bfloat16*)out_k,
                          (__nv_bfloat16*)out_v, status);
}

cudaError_t launch_compact_kept(const void* k, const void* v, long long stride_tok,
                                long long stride_head, const ReqTable& reqs, int n_kv_heads,
                                long long total_kept_rows, const int* kept_idx, int varlen_output,
                                long long out_stride_head, void* out_k, void* out_v, int* status,
                                cudaStream_t stream) {
    if (total_kept_rows <= 0) return cudaSuccess;
    const long long blocks = (total_kept_rows + 7) / 8;
    return launch_chained(compact_kept_kernel, dim3((unsigned)blocks), dim3(256), 0, stream,
                          (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, stride_tok, stride_head, reqs,
                          n_kv_heads, total_kept_rows, kept_idx, varlen_output, out_stride_head,
                          (__nv_bfloat16*)out_k, (__nv_bfloat16*)out_v, status);
}

cudaError_t launch_argmax_rows(const float* sim_matrix, const ReqTable& reqs,
                                    int n_kv_heads, int max_evicted, int* assign, float* sim,
                                    cudaStream_t stream) {
    if (max_evicted <= 0) return cudaSuccess;
    dim3 grid((max_evicted + 7) / 8, n_kv_heads, reqs.n);
    argmax_rows_kernel<<<grid, 256, 0, stream>>>(sim_matrix, reqs, n_kv_heads, assign, sim);
    return cudaGetLastError();
}

}  // namespace lookm
