// Exact FP32 re-rank of the candidate lists.
//
// Candidate selection (FP32 expansion form or BF16 tensor cores) only has to
// bring the true k nearest into each query's candidate set; this pass
// re-scores every candidate by direct difference, sum_t (x_t - y_t)^2 in FP32
// (no cancellation against |x|^2 + |y|^2), and orders by (distance, id), the
// exact-kNN definition with ties broken by index.  Cosine rows arrive
// normalised, so 1 - cos = |x^ - y^|^2 / 2 (paper, Methods, "Custom GPU
// kernels", defines both distances).
#include <math.h>
#include <limits.h>

#include "common.cuh"
#include "kernels.h"
#include "rerank.cuh"
#include "warp_sort.cuh"

namespace rsc {

namespace {

constexpr int kWarps = 16;   // queries per block: neighbouring queries share candidate rows in L1

// Every candidate of the kernels below comes through here: list entry jp names
// a position (its row in R, or perm's) when it lies in [0, n).  Empty entries
// and what a search that gave up left in the lists do not: -1, id INT_MAX.
__device__ __forceinline__ int candidate_row(int32_t jp, int64_t n, const int32_t *perm, bool r_by_pos, int &id) {
    id = INT_MAX;
    if (jp < 0 || (int64_t)jp >= n) return -1;
    id = perm ? perm[jp] : jp;   // original id
    return r_by_pos ? jp : id;
}

// Warp per query, 8 lanes per candidate row.  In step g, lanes 8 r + s
// (r < 4, s < 8) score candidate 4 g + r of the current 32 (rerank.cuh: eight
// components per lane, an FMA chain over them, three xor shuffles);
// candidate c's sum then goes to lane c % 32.  One load
// instruction of the warp touches 4 candidate rows instead of 32 (a lane per
// row): the gathers are bound by the L1's line lookups, not by bytes.
// E = (candidate slots rounded up to a power of two) / 32 (key, id) pairs per
// lane, element v = e * 32 + lane, sorted ascending by (key, id) with a
// bitonic network held in registers.  Up to 64 candidates fit in 32 registers
// a thread, so four blocks (all 64 warps) stay resident to hide the gathers'
// latency.
template <int E>
__global__ void __launch_bounds__(kWarps * 32, E <= 2 ? 4 : 1)
rerank_kernel(const float *__restrict__ R, int64_t rs, int64_t n, int d, int metric, bool vec,
              const int32_t *__restrict__ cand, int KC, int C, int k, const int32_t *__restrict__ perm,
              bool r_by_pos, int32_t *__restrict__ idx, float *__restrict__ dist) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 3, s = lane & 7;

    const int64_t q = (int64_t)blockIdx.x * kWarps + warp;   // position in the candidate lists
    if (q >= n) return;                                        // warp-uniform
    const int64_t qo = perm ? (int64_t)perm[q] : q;            // original row
    const int64_t qr = r_by_pos ? q : qo;                      // its row in R
    const bool cosine = metric == RSC_COSINE;

    float xv[8];
    rr::load8(R + qr * rs, s, d, cosine, vec, xv);
    const bool fq = cosine && R[qr * rs + d] != 0.f;

    float key[E];
    int id[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = e * 32 + lane;
        int row = -1;   // this lane's candidate: its row in R, -1 for none
        id[e] = INT_MAX;
        if (c < C) {
            const int sp = c / KC, slot = c - sp * KC;
            row = candidate_row(cand[((int64_t)sp * n + q) * KC + slot], n, perm, r_by_pos, id[e]);
        }
        key[e] = INFINITY;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            // an empty slot scores row 0 and is dropped below (no branch)
            const int yr = max(__shfl_sync(0xffffffffu, row, 4 * g + r), 0);
            float yv[8];
            rr::load8(R + (int64_t)yr * rs, s, d, cosine, vec, yv);
            const float part = rr::dist2(xv, yv);
            const float got = __shfl_sync(0xffffffffu, part, 8 * (lane & 3));
            if ((lane >> 2) == g && row >= 0) key[e] = got;
        }
        if (cosine && row >= 0) {
            const bool fy = __ldg(R + (int64_t)row * rs + d) != 0.f;
            if (fq || fy) key[e] = (fq && fy) ? 0.f : 2.f;
        }
    }

    warp_sort_pairs<E>(key, id);

#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = e * 32 + lane;
        if (c < k) {
            const bool valid = id[e] != INT_MAX;
            idx[qo * k + c] = valid ? id[e] : -1;
            dist[qo * k + c] = valid ? (cosine ? 0.5f * key[e] : sqrtf(key[e])) : INFINITY;
        }
    }
}

// More than 64 candidates, k <= 32: the same scores, 32 candidates at a time,
// each batch sorted and merged into the best 32, so that a lane holds one
// candidate and not C / 32 of them and three blocks stay resident whatever C is
// (128 candidates, k = 30, 400k rows: 2.40 ms with four pairs per lane and
// 58 registers, 1.75 ms so; 64 candidates are as fast as two pairs per lane).
__global__ void __launch_bounds__(kWarps * 32, 3)
rerank_stream_kernel(const float *__restrict__ R, int64_t rs, int64_t n, int d, int metric, bool vec,
                     const int32_t *__restrict__ cand, int KC, int C, int k, const int32_t *__restrict__ perm,
                     bool r_by_pos, int32_t *__restrict__ idx, float *__restrict__ dist) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 3, s = lane & 7;
    const int64_t q = (int64_t)blockIdx.x * kWarps + warp;   // position in the candidate lists
    if (q >= n) return;
    const int64_t qo = perm ? (int64_t)perm[q] : q;            // original row
    const int64_t qr = r_by_pos ? q : qo;                      // its row in R
    const bool cosine = metric == RSC_COSINE;
    float xv[8];
    rr::load8(R + qr * rs, s, d, cosine, vec, xv);
    const bool fq = cosine && R[qr * rs + d] != 0.f;
    float bk[1] = {INFINITY};   // the best 32, ascending over the lanes
    int bi[1] = {INT_MAX};
#pragma unroll 1
    for (int c0 = 0; c0 < C; c0 += 32) {
        const int c = c0 + lane;
        int row = -1;   // this lane's candidate: its row in R, -1 for none
        float key[1] = {INFINITY};
        int id[1] = {INT_MAX};
        if (c < C) {
            const int sp = c / KC, slot = c - sp * KC;
            row = candidate_row(cand[((int64_t)sp * n + q) * KC + slot], n, perm, r_by_pos, id[0]);
        }
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            // an empty slot scores row 0 and is dropped below (no branch)
            const int yr = max(__shfl_sync(0xffffffffu, row, 4 * g + r), 0);
            float yv[8];
            rr::load8(R + (int64_t)yr * rs, s, d, cosine, vec, yv);
            const float part = rr::dist2(xv, yv);
            const float got = __shfl_sync(0xffffffffu, part, 8 * (lane & 3));
            if ((lane >> 2) == g && row >= 0) key[0] = got;
        }
        if (cosine && row >= 0) {
            const bool fy = __ldg(R + (int64_t)row * rs + d) != 0.f;
            if (fq || fy) key[0] = (fq && fy) ? 0.f : 2.f;
        }
        warp_sort_pairs<1>(key, id);
        if (c0 == 0) {
            bk[0] = key[0];
            bi[0] = id[0];
        } else {
            warp_merge_best(bk[0], bi[0], key[0], id[0]);
        }
    }
    if (lane < k) {
        const bool valid = bi[0] != INT_MAX;
        idx[qo * k + lane] = valid ? bi[0] : -1;
        dist[qo * k + lane] = valid ? (cosine ? 0.5f * bk[0] : sqrtf(bk[0])) : INFINITY;
    }
}

// Re-rank from the parts' lists, warp per query: the k-th smallest key (by
// bisection on the keys' ordered bits, E per lane; a few more than k below the
// final bound do no harm) bounds what can be among the k nearest, the ids
// within its reach (k and a few) are compacted into shared memory, scored as in
// rerank_kernel, 32 at a time, and merged into the best 32.  A row with more
// than kMax of them, or with a list that may have left some out, goes to the
// ties pass.  10,000 rows, k = 15: 7 parts, 168 candidates a row, 22 us (256 of
// eight splits before, all scored: 267 us).
template <int E>
__global__ void __launch_bounds__(kWarps * 32)
rerank_parts_kernel(const float *__restrict__ R, int64_t rs, int64_t n, int d, int metric, bool vec, SimtParts P,
                    int width, int k, int32_t *__restrict__ idx, float *__restrict__ dist) {
    constexpr int kMax = 64;
    __shared__ int32_t ids_s[kWarps][kMax];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = lane >> 3, s = lane & 7;
    const int64_t q = (int64_t)blockIdx.x * kWarps + warp;
    if (q >= n) return;
    int32_t *ids = ids_s[warp];
    const int M = P.segs * P.list;
    const float *pk = P.key + q * M;
    const int32_t *pi = P.id + q * M;
    // unsigned bits that order as the floats do
    auto order = [](float f) {
        const unsigned u = __float_as_uint(f);
        return u & 0x80000000u ? ~u : u | 0x80000000u;
    };
    unsigned key[E];
    int32_t id[E];
    unsigned lo = 0xffffffffu;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int c = e * 32 + lane;
        int unused;
        id[e] = c < M ? candidate_row(pi[c], n, nullptr, false, unused) : -1;
        key[e] = id[e] >= 0 ? order(pk[c]) : 0xffffffffu;
        lo = min(lo, key[e]);
    }
    // k keys lie at or below the k-th of any list: the smallest of these
    unsigned hi = lane < P.segs && pi[lane * P.list + k - 1] >= 0 ? order(pk[lane * P.list + k - 1]) : 0xffffffffu;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_min_sync(0xffffffffu, hi);
    while (lo < hi) {   // smallest bound with at least k keys at or below it (stops early when it is exactly k)
        const unsigned mid = lo + (hi - lo) / 2;
        int c = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) c += key[e] <= mid ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= k) hi = mid;
        else lo = mid + 1;
        if (c == k) break;
    }
    // fewer than k rows: hi stays at the top and everything is scored
    const float vv = P.vv[q];
    const float t = hi == 0xffffffffu ? INFINITY : __uint_as_float(hi & 0x80000000u ? hi & 0x7fffffffu : ~hi);
    float reach = hi == 0xffffffffu ? INFINITY : rr::reach(t, vv, sqrtf(vv), width);
    if (!(reach < INFINITY)) reach = INFINITY;
    const unsigned within = order(reach);
    int count = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool in = id[e] >= 0 && key[e] <= within;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        const int at = count + __popc(m & ((1u << lane) - 1u));
        if (in && at < kMax) ids[at] = id[e];
        count += __popc(m);
    }
    // a full list whose last entry is within reach may have left some out
    const bool cut = lane < P.segs && pi[lane * P.list + P.list - 1] >= 0 &&
                     order(pk[lane * P.list + P.list - 1]) <= within;
    const bool tie = __any_sync(0xffffffffu, cut) || count > kMax;
    if (lane == 0) {
        P.tie_bound[q] = tie ? reach : -INFINITY;
        if (tie && atomicExch(P.tie_flag + q / kTieItem, 1) == 0)
            P.tie_items[atomicAdd(P.tie_count, 1)] = (int32_t)(q / kTieItem);
    }
    if (tie) return;
    __syncwarp();
    const bool cosine = metric == RSC_COSINE;
    float xv[8];
    rr::load8(R + q * rs, s, d, cosine, vec, xv);
    const bool fq = cosine && R[q * rs + d] != 0.f;
    float bk[1] = {INFINITY};   // the best 32, ascending over the lanes
    int bi[1] = {INT_MAX};
    for (int c0 = 0; c0 < count; c0 += 32) {
        const int row = c0 + lane < count ? ids[c0 + lane] : -1;
        float ck[1] = {INFINITY};
        int ci[1] = {row >= 0 ? row : INT_MAX};
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            if (c0 + 4 * g >= count) break;   // warp-uniform
            const int yr = max(__shfl_sync(0xffffffffu, row, 4 * g + r), 0);
            float yv[8];
            rr::load8(R + (int64_t)yr * rs, s, d, cosine, vec, yv);
            const float part = rr::dist2(xv, yv);
            const float got = __shfl_sync(0xffffffffu, part, 8 * (lane & 3));
            if ((lane >> 2) == g && row >= 0) ck[0] = got;
        }
        if (cosine && row >= 0) {
            const bool fy = __ldg(R + (int64_t)row * rs + d) != 0.f;
            if (fq || fy) ck[0] = (fq && fy) ? 0.f : 2.f;
        }
        warp_sort_pairs<1>(ck, ci);
        if (c0 == 0) {
            bk[0] = ck[0];
            bi[0] = ci[0];
        } else {
            warp_merge_best(bk[0], bi[0], ck[0], ci[0]);
        }
    }
    if (lane < k) {
        const bool valid = bi[0] != INT_MAX;
        idx[q * k + lane] = valid ? bi[0] : -1;
        dist[q * k + lane] = valid ? (cosine ? 0.5f * bk[0] : sqrtf(bk[0])) : INFINITY;
    }
}

// dst row i <- src row perm[i] (width floats, zero-padded to dst_stride, a
// multiple of 4 with a 16-byte aligned dst); 16 lanes per row, a float4 store
// per lane and step.
__global__ void gather_rows_kernel(const float *__restrict__ src, int64_t src_stride, int64_t n, int width,
                                   const int32_t *__restrict__ perm, float *__restrict__ dst, int64_t dst_stride) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    const int l = threadIdx.x & 15;
    if (i >= n) return;
    const float *s = src + (int64_t)perm[i] * src_stride;
    float4 *o = reinterpret_cast<float4 *>(dst + i * dst_stride);
    for (int f = l; 4 * f < dst_stride; f += 16) {
        const int t = 4 * f;
        o[f] = make_float4(t < width ? s[t] : 0.f, t + 1 < width ? s[t + 1] : 0.f, t + 2 < width ? s[t + 2] : 0.f,
                           t + 3 < width ? s[t + 3] : 0.f);
    }
}

}  // namespace

cudaError_t launch_gather_rows(const float *src, int64_t src_stride, int64_t n, int width, const int32_t *perm,
                               float *dst, int64_t dst_stride, cudaStream_t st) {
    if (dst_stride % 4 != 0 || reinterpret_cast<uintptr_t>(dst) % 16 != 0) return cudaErrorInvalidValue;
    gather_rows_kernel<<<(unsigned)ceil_div(n * 16, 256), 256, 0, st>>>(src, src_stride, n, width, perm, dst,
                                                                      dst_stride);
    return cudaGetLastError();
}

cudaError_t launch_rerank_parts(const float *R, int64_t rs, int64_t n, int d, int metric, const SimtParts &parts,
                                int width, int k, int32_t *idx, float *dist, cudaStream_t st) {
    const int M = parts.segs * parts.list;
    const bool vec = rs % 4 == 0 && reinterpret_cast<uintptr_t>(R) % 16 == 0;
    auto kern = M <= 6 * 32 ? rerank_parts_kernel<6> : M <= 12 * 32 ? rerank_parts_kernel<12> : rerank_parts_kernel<20>;
    if (M > 20 * 32 || k > 32 || k > parts.list) return cudaErrorInvalidValue;
    kern<<<(unsigned)ceil_div(n, kWarps), kWarps * 32, 0, st>>>(R, rs, n, d, metric, vec, parts, width, k, idx, dist);
    return cudaGetLastError();
}

cudaError_t launch_rerank(const float *R, int64_t rs, int64_t n, int d, int metric,
                          const int32_t *cand, int KC, int splits, int k, const int32_t *perm, bool r_by_pos,
                          int32_t *idx, float *dist, cudaStream_t st) {
    const int C = KC * splits;
    int C2 = 32;
    while (C2 < C) C2 <<= 1;
    if (C2 > 1024 || k > C) return cudaErrorInvalidValue;
    const unsigned blocks = (unsigned)ceil_div(n, kWarps);
    if (d < 1 || d > 64) return cudaErrorInvalidValue;   // 8 lanes x 8 components per row
    // vector loads when every row starts on a 16-byte boundary
    const bool vec = rs % 4 == 0 && reinterpret_cast<uintptr_t>(R) % 16 == 0;
    if (C > 64 && k <= 32) {
        rerank_stream_kernel<<<blocks, kWarps * 32, 0, st>>>(R, rs, n, d, metric, vec, cand, KC, C, k, perm, r_by_pos,
                                                             idx, dist);
        return cudaGetLastError();
    }
#define RSC_RR(e)                                                                                                    \
    case 32 * e:                                                                                                     \
        rerank_kernel<e><<<blocks, kWarps * 32, 0, st>>>(R, rs, n, d, metric, vec, cand, KC, C, k, perm, r_by_pos, \
                                                         idx, dist);                                                 \
        break
    switch (C2) {
        RSC_RR(1); RSC_RR(2); RSC_RR(4); RSC_RR(8); RSC_RR(16); RSC_RR(32);
        default: return cudaErrorInvalidValue;
    }
#undef RSC_RR
    return cudaGetLastError();
}

}  // namespace rsc
