// Selection kernel: recent window, text prior and Top-N (Eq. 5-8), one CTA per (request, KV head).
//
// The text prior is applied as an ordering rule: adding T_p = max(A_s) to every text score makes
// any text token outrank any image token (scores are positive), so candidates are ordered by
// (is_text, score, lower position).  With n_text text candidates and N slots:
//   n_text <= N : all text candidates are kept and the best N - n_text image candidates;
//   n_text >  N : the best N text candidates are kept and no image candidate.
// Without a mask (text prior off: Eq. 8 on the raw scores) every candidate is in the text class,
// which reduces to a plain Top-N by score.
// Either way one class is kept wholesale or not at all and the other needs an exact top-k.  The k-th
// largest key (order-preserving 32-bit image of the score) is found by bisection between the smallest
// and the largest one: a step counts the keys at or above the middle, with the keys in registers and
// one block barrier.  (Prompts too long for the registers count 2048 parts of that range instead, see
// select_kernel.)  Ties at the threshold go to the lowest positions.  An ordered pass over the same
// registers writes the kept and evicted lists in ascending position: ballots number a warp's tokens, one
// block scan the warps.
//
// The kernel is bound by the latency of one CTA's barriers and round trips.  A four-pass radix select
// over a shared-memory histogram (its first digits nearly equal for all scores, so that the atomics
// collide), two block scans and a second reading of the scores for the lists | this, lookm_select with 32
// heads, us: 2048 tokens 14.4 | 8.9, 8192 18.4 | 15.0, 16384 30.7 | 25.4, 32768 55 | 44, 65536 122 | 89, 262144 513 | 386.
//
// The selection occupies only n_requests * n_kv_heads CTAs, so the same launch carries, in further
// CTAs, work that does not depend on it and is needed next: 1 / |k| of every key row (the cosine
// denominators of Eq. 9).
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"

namespace lookm {
namespace {

__device__ __forceinline__ unsigned order_key(float s) {
    unsigned b = __float_as_uint(s);
    if (b == 0x80000000u) b = 0u;                        // -0 and +0 compare equal
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);   // larger float <=> larger key
}

// Sums of two ints per warp over the warps before the caller's, and over all (ta, tb).
template <int kThreads>
__device__ __forceinline__ void warp_scan2(int a, int b, int& ea, int& eb, int& ta, int& tb, int (*warp_tot)[2]) {
    constexpr int kWarps = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();                                     // protects warp_tot from the previous use
    if (lane == 0) { warp_tot[warp][0] = a; warp_tot[warp][1] = b; }
    __syncthreads();
    const int wa = lane < kWarps ? warp_tot[lane][0] : 0, wb = lane < kWarps ? warp_tot[lane][1] : 0;
    ta = __reduce_add_sync(0xffffffffu, wa);
    tb = __reduce_add_sync(0xffffffffu, wb);
    ea = __reduce_add_sync(0xffffffffu, lane < warp ? wa : 0);
    eb = __reduce_add_sync(0xffffffffu, lane < warp ? wb : 0);
}

// A lane's share of |row|^2: the squares of its eight elements.
__device__ __forceinline__ float sum_squares(const uint4& u) {
    const unsigned w[4] = {u.x, u.y, u.z, u.w};
    float ss = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float lo = __uint_as_float(w[j] << 16), hi = __uint_as_float(w[j] & 0xffff0000u);
        ss = fmaf(lo, lo, ss);
        ss = fmaf(hi, hi, ss);
    }
    return ss;
}

// 1 / |k| of every key row (0 for a zero row): half a warp per row, 16 bytes per lane, four rows
// in flight per half-warp (the loop is bound by memory latency otherwise).  Row r is token
// r / n_kv_heads of head r % n_kv_heads; quotient, remainder and address are carried along instead of
// computed every time.  The four rows are added up together, each ending in a quarter of the half-warp,
// so that one root and one division serve all of them (with four sums over the half-warp and four of
// these the loop is bound by instructions; the launch takes then | now 28.6 us | 20.5 with 8192 tokens x 32
// heads, 66.6 | 49.6 with 16384 x 40).
template <int kThreads>
__device__ __forceinline__ void key_norms(const __nv_bfloat16* __restrict__ k, long long stride_tok,
                                          long long stride_head, int n_kv_heads, long long T,
                                          float* __restrict__ rnorm_all, int block, int n_blocks) {
    constexpr int kRowsPerBlock = kThreads / 16;
    const int half = threadIdx.x >> 4, l16 = threadIdx.x & 15;
    const long long n_rows = T * n_kv_heads;
    const long long step = (long long)n_blocks * kRowsPerBlock;      // rows between two of my rows
    const long long step_tok = step / n_kv_heads;
    const int step_h = (int)(step % n_kv_heads);
    const long long step_at = step_tok * stride_tok + step_h * stride_head, wrap_at = stride_tok - n_kv_heads * stride_head;
    const long long step_out = step_h * T + step_tok, wrap_out = 1 - n_kv_heads * T;
    long long r = (long long)block * kRowsPerBlock + half;
    const long long tok = r / n_kv_heads;
    int h = (int)(r % n_kv_heads);
    const __nv_bfloat16* at = k + tok * stride_tok + h * stride_head + l16 * 8;
    long long out = h * T + tok;
    const bool bit8 = l16 & 8, bit4 = l16 & 4;
    // the loop bound is the warp's first row, so that both half-warps always reach the shuffles
    for (long long rw = r - (half & 1); rw < n_rows; rw += 4 * step) {
        uint4 u[4];
        long long mine = -1;                             // where this lane's quarter's row goes
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            u[i] = make_uint4(0u, 0u, 0u, 0u);
            if (r < n_rows) {
                u[i] = *reinterpret_cast<const uint4*>(at);
                if (l16 == i * 4) mine = out;
            }
            r += step;
            at += step_at;
            out += step_out;
            h += step_h;
            if (h >= n_kv_heads) { h -= n_kv_heads; at += wrap_at; out += wrap_out; }
        }
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = sum_squares(u[i]);
        // lanes with bit 8 take rows 2 and 3, of these lanes with bit 4 rows 1 and 3
#pragma unroll
        for (int i = 0; i < 2; ++i)
            x[i] = (bit8 ? x[i + 2] : x[i]) + __shfl_xor_sync(0xffffffffu, bit8 ? x[i] : x[i + 2], 8, 16);
        float ss = (bit4 ? x[1] : x[0]) + __shfl_xor_sync(0xffffffffu, bit4 ? x[0] : x[1], 4, 16);
        ss += __shfl_xor_sync(0xffffffffu, ss, 2, 16);
        ss += __shfl_xor_sync(0xffffffffu, ss, 1, 16);
        if (mine >= 0) rnorm_all[mine] = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
    }
}

// The first kThreads * kSteps tokens are shared out evenly: a warp has steps * 32 consecutive ones, a step
// is one per lane, and their keys stay in registers.  kLong: there may be tokens beyond, which every pass has
// to read again.  Then a pass counts 2048 parts of the range between the smallest and the largest key, and
// goes on in the one that holds the k-th largest: three passes where the bisection takes some 27.
constexpr int kParts = 2048;
template <int kThreads, int kSteps, bool kLong>
__global__ void __launch_bounds__(kThreads)
select_kernel(const float* __restrict__ scores, const uint8_t* __restrict__ mask,
              const Req* __restrict__ reqs, int n_select_blocks, int n_kv_heads, long long T,
              int* __restrict__ kept_idx, int* __restrict__ evict_idx, int* __restrict__ rank,
              const __nv_bfloat16* __restrict__ keys, long long stride_tok, long long stride_head,
              float* __restrict__ rnorm_all) {
    constexpr int kWarps = kThreads / 32, kChunk = kThreads * kSteps;
    static_assert(kSteps % 8 == 0 && kSteps <= 32, "steps are skipped by eights; a bit per step");
    __shared__ int warp_tot[kWarps][2];
    __shared__ int counts[2][32];
    __shared__ unsigned extremes[2][32];

    grid_dependency_wait();
    if ((int)blockIdx.x >= n_select_blocks) {
        key_norms<kThreads>(keys, stride_tok, stride_head, n_kv_heads, T, rnorm_all, (int)blockIdx.x - n_select_blocks,
                            (int)gridDim.x - n_select_blocks);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // (from the table, also of a single prompt: by value 700 tokens x 32 heads 8.7 | 9.5 us, 131072 x 8 187.3 | 189,
    // a layer of 700 x 32 52.7 either way)
    const Req rq = reqs[blockIdx.x / n_kv_heads];
    const int h = blockIdx.x % n_kv_heads;
    const float* s = scores + (long long)h * T + rq.tok_begin;
    const uint8_t* msk = mask ? mask + rq.tok_begin : nullptr;
    auto is_image = [msk](int j) { return msk != nullptr && msk[j] != 0; };
    const int L = rq.L, B = rq.B, M = rq.M;
    const int N = B - M, nc = L - M;                     // slots to fill, candidates (the rest is the window)
    int turn = 0;                                        // alternates the buffers of block_sum
    auto block_sum = [&](int x) {
        x = __reduce_add_sync(0xffffffffu, x);
        if (lane == 0) counts[turn][warp] = x;
        __syncthreads();
        x = __reduce_add_sync(0xffffffffu, lane < kWarps ? counts[turn][lane] : 0);
        turn ^= 1;
        return x;
    };

    // ---- keys and classes of this thread's tokens --------------------------------------------------
    const int steps = min(kSteps, (L + kThreads - 1) / kThreads);
    const int first = warp * steps * 32 + lane;          // token of step q: first + 32 q
    unsigned key[kSteps];
    unsigned img = 0u;                                   // bit q: candidate of step q is an image token
    auto load = [&](int j0) {
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            const int j = j0 + q * 32;
            key[q] = 0u;
            if (q < steps && j < nc) {
                key[q] = order_key(s[j]);
                img |= (is_image(j) ? 1u : 0u) << q;
            }
        }
    };
    load(first);
    // the candidates beyond, with the loads of eight in flight together
    constexpr int kBatch = 8;
    auto beyond = [&](auto visit) {
        for (int j0 = kChunk + threadIdx.x; kLong && j0 < nc; j0 += kBatch * kThreads) {
            float v[kBatch];
            bool image[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const int j = j0 + q * kThreads;
                v[q] = j < nc ? s[j] : 0.f;
                image[q] = j < nc && is_image(j);
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q)
                if (j0 + q * kThreads < nc) visit(order_key(v[q]), image[q]);
        }
    };
    // text candidates: candidates less image tokens among them
    int cnt = min(steps, max(0, (nc - first + 31) / 32)) - __popc(img);
    beyond([&](unsigned, bool image) { cnt += !image; });
    const int n_text = block_sum(cnt);
    // class whose members are ranked (1 = image); the other class is kept entirely or not at all
    const int sel_cls = (n_text <= N) ? 1 : 0;
    const bool other_kept = (n_text <= N);
    const int k = (n_text <= N) ? (N - n_text) : N;      // how many of sel_cls to keep
    const int n_sel = sel_cls ? (nc - n_text) : n_text;
    const bool take_all = (k >= n_sel), take_none = (k <= 0);

    // ---- key of the k-th largest member of sel_cls -------------------------------------------------
    unsigned thr = 0u;          // members above thr are kept ...
    int need_ties = 0;          // ... and so many of those equal to it (lowest positions first)
    if (!take_all && !take_none) {
        // members keep their key, everything else gets 0 (no finite score maps to it)
        unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            const bool member = q < steps && first + q * 32 < nc && ((img >> q) & 1u) == (unsigned)sel_cls;
            if (!member) key[q] = 0u;
            if (member) { lo = min(lo, key[q]); hi = max(hi, key[q]); }
        }
        beyond([&](unsigned x, bool image) { if (image == (sel_cls != 0)) { lo = min(lo, x); hi = max(hi, x); } });
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) { extremes[0][warp] = lo; extremes[1][warp] = hi; }
        __syncthreads();
        lo = __reduce_min_sync(0xffffffffu, lane < kWarps ? extremes[0][lane] : 0xffffffffu);
        hi = __reduce_max_sync(0xffffffffu, lane < kWarps ? extremes[1][lane] : 0u);
        if (kLong) {
            __shared__ int parts[kParts], found[2];
            need_ties = k;                               // of those left in [lo, hi]
            while (lo < hi) {
                const int shift = max(0, 32 - __clz(hi - lo) - 11);
                for (int i = threadIdx.x; i < kParts; i += kThreads) parts[i] = 0;
                __syncthreads();
                auto count = [&](unsigned x) { if (x >= lo && x <= hi) atomicAdd(&parts[(x - lo) >> shift], 1); };
#pragma unroll
                for (int q = 0; q < kSteps; ++q)
                    if (q < steps && first + q * 32 < nc && ((img >> q) & 1u) == (unsigned)sel_cls) count(key[q]);
                beyond([&](unsigned x, bool image) { if (image == (sel_cls != 0)) count(x); });
                __syncthreads();
                // parts from the top, kOwn per thread: the one in which the count reaches need_ties
                constexpr int kOwn = kParts / kThreads;
                int c[kOwn], mine = 0, before, other, all, none;
#pragma unroll
                for (int q = 0; q < kOwn; ++q) mine += c[q] = parts[kParts - 1 - (int)threadIdx.x * kOwn - q];
                int incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += x;
                }
                warp_scan2<kThreads>(__shfl_sync(0xffffffffu, incl, 31), 0, before, other, all, none, warp_tot);
                before += incl - mine;
#pragma unroll
                for (int q = 0; q < kOwn; ++q) {
                    if (before < need_ties && before + c[q] >= need_ties) {
                        found[0] = kParts - 1 - (int)threadIdx.x * kOwn - q;
                        found[1] = need_ties - before;
                    }
                    before += c[q];
                }
                __syncthreads();
                lo += (unsigned)found[0] << shift;
                if (hi - lo > (1u << shift) - 1u) hi = lo + ((1u << shift) - 1u);
                need_ties = found[1];
            }
            thr = lo;
        } else {
            int above = 0;                               // members above hi
            bool exact = false;
            while (lo < hi && !exact) {                  // at least k members >= lo, fewer than k above hi
                const unsigned mid = lo + (hi - lo) / 2u + 1u;
                int c = 0;
#pragma unroll
                for (int g = 0; g < kSteps; g += 8)
                    if (g < steps)
#pragma unroll
                        for (int q = g; q < g + 8; ++q) c += key[q] >= mid;
                c = block_sum(c);
                if (c == k) { thr = mid - 1u; exact = true; }
                else if (c > k) lo = mid;
                else { hi = mid - 1u; above = c; }
            }
            if (!exact) { thr = lo; need_ties = k - above; }
        }
    }

    // ---- ordered emission -----------------------------------------------------------------------
    const long long kept_base = rq.kept_off + (long long)h * B;
    const long long ev_base = rq.ev_off + (long long)h * rq.E;
    int* rk = rank ? rank + (long long)h * T + rq.tok_begin : nullptr;
    const unsigned lt_mask = (1u << lane) - 1u;
    int kept_run = 0, tie_run = 0;
    for (int c0 = 0; c0 < (kLong ? L : 1); c0 += kChunk) {       // (steps == kSteps if there is more than one turn)
        const int j0 = c0 + first;
        if (kLong && c0) { img = 0u; load(j0); }
        unsigned keep = 0u, tie = 0u;                    // bit q: token of step q
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            const int j = j0 + q * 32;
            if (q >= steps || j >= L) continue;
            if (j >= nc) keep |= 1u << q;
            else if (((img >> q) & 1u) != (unsigned)sel_cls) keep |= (other_kept ? 1u : 0u) << q;
            else if (take_all) keep |= 1u << q;
            else if (!take_none) {
                if (key[q] > thr) keep |= 1u << q;
                else if (key[q] == thr) tie |= 1u << q;
            }
        }
        // a tie is kept while fewer than need_ties equal keys precede it, so the kept ones before a
        // token are the sure ones before it and min(need_ties, ties before it)
        int sure, ties, t_keep, t_tie;
        warp_scan2<kThreads>(__reduce_add_sync(0xffffffffu, __popc(keep)), __reduce_add_sync(0xffffffffu, __popc(tie)), sure, ties,
                             t_keep, t_tie, warp_tot);
        sure += kept_run;
        ties += tie_run;
#pragma unroll
        for (int q = 0; q < kSteps; ++q) {
            if (q >= steps) continue;
            const int j = j0 + q * 32;
            const bool is_keep = (keep >> q) & 1u, is_tie = (tie >> q) & 1u;
            const unsigned keeps = __ballot_sync(0xffffffffu, is_keep), tied = __ballot_sync(0xffffffffu, is_tie);
            const int before = ties + __popc(tied & lt_mask);
            const int slot = sure + __popc(keeps & lt_mask) + min(need_ties, before);
            if (j < L) {
                if (is_keep || (is_tie && before < need_ties)) {
                    kept_idx[kept_base + slot] = j;
                    if (rk) rk[j] = -1 - slot;
                } else {
                    const int e = j - slot;              // evicted before j = j - kept before j
                    evict_idx[ev_base + e] = j;
                    if (rk) rk[j] = e;
                }
            }
            sure += __popc(keeps);
            ties += __popc(tied);
        }
        kept_run += t_keep;
        tie_run += t_tie;
    }
}

}  // namespace

cudaError_t launch_select(const float* scores, const uint8_t* mask, const ReqTable& reqs,
                          int n_kv_heads, long long T, int max_L, int* kept_idx, int* evict_idx, int* rank,
                          const void* k_for_norms, long long stride_tok, long long stride_head,
                          float* rnorm_all, int num_sms, cudaStream_t stream) {
    const int n_select = n_kv_heads * reqs.n;
    // Cheaper barriers with fewer threads, a shorter chain of steps with more: a layer of 2048 tokens x 8
    // heads takes 67.0 us with 256 threads, 64.9 with 512 and 65.8 with 1024, 2048 x 32 123, 119.5 and
    // 119.5, 3000 x 8 85.1 with 512 and 84.2 with 1024.  Registers hold up to 32768 tokens, in variants of 8, 16 and
    // 32 per thread (the last spills: 16384 tokens x 8 heads 32.8 us with 32, 21.3 with 16); beyond, sixteen are
    // held and the rest is read again (65536 tokens x 8 heads 88 us; bisected with 32 held 179).
    typedef void (*Kernel)(const float*, const uint8_t*, const Req*, int, int, long long, int*, int*, int*, const __nv_bfloat16*,
                           long long, long long, float*);
    struct Variant { int threads, most; Kernel kernel; };
    static const Variant variants[] = {{512, 512 * 4, select_kernel<512, 8, false>}, {1024, 1024 * 8, select_kernel<1024, 8, false>},
                                       {1024, 1024 * 16, select_kernel<1024, 16, false>}, {1024, 1024 * 32, select_kernel<1024, 32, false>},
                                       {1024, 0x7fffffff, select_kernel<1024, 16, true>}};
    const Variant* use = variants;
    while (max_L > use->most) ++use;
    const int threads = use->threads;
    int n_norm = 0;
    if (k_for_norms) {
        // the norm CTAs take the SMs that the selection leaves free, so that all of them run at once
        // (a second wave would have to wait for the selection CTAs, which run longest)
        const long long want = (T * n_kv_heads + threads / 16 - 1) / (threads / 16);
        const int per_sm = 1024 / threads;
        // (with selection CTAs on more than half of the SMs the few SMs left would carry all the
        // norms: then a full wave of norm CTAs follows the selection CTAs instead)
        n_norm = (int)std::min<long long>(want, (long long)per_sm * (n_select < num_sms / 2 ? num_sms - n_select : num_sms));
    }
    return launch_chained(use->kernel, dim3(n_select + n_norm), dim3(threads), 0, stream,
                          scores, mask, reqs.rows, n_select, n_kv_heads, T, kept_idx, evict_idx, rank,
                          (const __nv_bfloat16*)k_for_norms, stride_tok, stride_head, rnorm_all);
}

}  // namespace lookm
