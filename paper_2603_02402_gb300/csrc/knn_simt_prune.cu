// FP32 SIMT candidate search on rows in locality order, with exact tile
// pruning (the plain-precision path of larger inputs).
//
// The full scan of knn_simt.cuh does n^2 distances.  On ordered rows almost
// all of them are of tiles that lie far away, and that can be shown from the
// tiles' bounding spheres, as in the tensor-core search (prune.cu): with
// s_ij = |y_j|^2 - 2 y_i.y_j = |y_i - y_j|^2 - |y_i|^2 (Euclidean; cosine rows:
// beta = 1 and |y_j|^2 left out of s), tile t cannot hold a neighbour of query
// tile Q when
//     (|c_Q - c_t| - r_Q - r_t)^2 - beta N_t - margin > tau_Q,
// tau_Q = max over Q's rows of (bound_i + |y_i|^2), margin = 2^-11 (N_Q + N_t)
// for the FP32 rounding of the bound itself, N = largest |y|^2 of a tile.
//
// bound_i is the row's current k-th smallest s plus twice e_i, a bound on how
// far a computed s_ij + |y_i|^2 and the re-rank's distance can differ:
//     e_i = 1.25 u (w + 20) (2 V (V + D) + (V + D)^2),   u = 2^-24,
// w the components of a row, V = |y_i|, D the distance of the k-th: the FMA
// chain errs by at most w u |y_i||y_j|, |y_j|^2 by (w + 1) u |y_j|^2, the
// re-rank's own sum by 12 u D^2, the rounding of the centred rows changes a
// squared distance by 2 u D (2 V + D), and |y_j| <= V + D for every row that
// matters.  Whatever lies above bound_i has
// a larger re-rank distance than k rows that are already in the list, so the
// k nearest are always among the kept ones and the result is that of the full
// scan.  Lists hold KC > k entries; a row whose list is full of entries within
// its bound (many rows at nearly the same distance as the k-th) is finished by
// ties_kernel, which scores every such row by the re-rank's own arithmetic.
//
// Tiles hold 64 consecutive rows, cut anew wherever two successive leaves of
// the ordering lie apart (the tile before is padded): a tile across such a gap
// spans two clusters, and its sphere keeps nearly every tile (100k rows, 60
// clusters, tiles cut every 64 rows whatever the leaves: 10.9 % of the pairs
// scanned and a few items that scanned everything, 15.4 ms).
//
// One persistent CTA pair per SM; an item is two tiles of query rows, each
// with its own sphere and tau (the database tile is scanned when either keeps
// it).  The CTA scans the tiles around its own, then walks the database in
// chunks of 256 tiles from its own chunk on: tests every tile's sphere against
// its current taus, and scans the tiles that are left.  A tile's record (64 rows transposed, then
// |y|^2) is one contiguous block, brought in by a bulk copy two tiles ahead.
// A thread accumulates an 8 x 8 block of (query, row) pairs by packed FP32
// fused multiply-adds (fma.rn.f32x2: two pairs per instruction, each rounded
// as the scalar one; half the issue slots), then scans its own query's row of
// the s tile with the register top-k.
//
// What bounds it: the FMA pipe and, next to it, the insertions (a row takes in
// about 70 values).  50 components, k = 15, one GB300, whole call (in brackets
// the full scan): 100,003 rows, 60 clusters 1.6 ms (25.9), of which this kernel
// 0.8 and the ordering 0.5; 1M rows, 100 clusters 31 ms (2054); rows without
// any clusters, of which no tile is dropped, 1.9 ms (1.5) at 16,384 rows, 9.1
// (7.3) at 50,000, 25.0 (25.9) at 100,003.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "rerank.cuh"
#include "tc_ptx.cuh"
#include "topk.cuh"

namespace rsc {

namespace simtp {

constexpr int kQ = 128;                   // query rows per item, threads per CTA
constexpr int kR = 64;                    // database rows per tile
constexpr int kPitch = kR + 4;            // s rows on 16 bytes, conflict-free scans
constexpr int kCap = 20;                  // top-k buffer entries per thread
constexpr int kChunk = 256;               // tiles tested at a time
constexpr int kWords = kChunk / 32;
constexpr int kSeeds = 8;                 // nearest tiles scanned first when the window's do not bound an item
constexpr int kWin = 3;                   // tiles on each side of the query tile scanned first
constexpr int kStages = 2;
constexpr int kMaxCtas = 320;             // persistent CTAs at most
constexpr int kBigItems = 192;            // items that may be split
constexpr int kSegs = 8;                  // parts of a split item at most
constexpr int kSegTiles = 128;            // tiles per part at least
constexpr uint32_t kSleepNs = 2000;                // suspend of a wait per try
constexpr long long kDrainBudget = 2000000000LL;   // ~1 s of SM clocks, for copies in flight when a CTA leaves

// tiles at most: every leaf may end in a partial one; an even number
__host__ __device__ inline int64_t tiles_max(int64_t n) { return (ceil_div(n, (int64_t)kR) + kOrderMaxLeaves + 2) / 2 * 2; }
// record of a tile: DP x 64 components, then 64 |y|^2
__host__ __device__ inline int record_floats(int DP) { return (DP + 1) * kR; }

struct Smem {
    int xs, ys, s, buf, list, cen, bars, total;   // byte offsets
};
__host__ __device__ inline Smem smem_layout(int DP) {
    Smem m;
    m.xs = 0;                                             // query tile: two records' components
    m.ys = m.xs + 2 * DP * kR * 4;
    m.s = m.ys + kStages * record_floats(DP) * 4;
    m.buf = m.s + kQ * kPitch * 4;
    m.list = m.buf + 2 * kCap * kQ * 4;
    m.cen = m.list + kChunk * 4;
    m.bars = m.cen + 2 * 64 * 4;
    m.total = m.bars + 256;
    return m;
}

// ------------------------------------------------------------------ packing

// The tiles: tile_pos[t] = first sorted position, tile_rows[t] = rows; *T =
// their number.  Successive leaves form a run unless their centroids are
// further apart than twice the sum of their mean squared radii; runs are cut
// into tiles of 64.  One block, two leaves (then two runs) per thread.
__global__ void __launch_bounds__(1024)
tile_table_kernel(const OrderLeaves lv, int64_t n, int DP, int32_t *__restrict__ tile_pos,
                  int32_t *__restrict__ tile_rows, int32_t *__restrict__ T) {
    static_assert(kOrderMaxLeaves <= 2048, "two leaves per thread");
    __shared__ int cid[2048], pos[2049], run_pos[2049], run_tile[2049];
    __shared__ int ws[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // exclusive scan of two values per thread; *total on every thread
    auto scan2 = [&](int c0, int c1, int *total) {
        int x = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        __syncthreads();
        if (lane == 31) ws[warp] = x;
        __syncthreads();
        int before = x - c0 - c1, all = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) before += ws[w];
            all += ws[w];
        }
        *total = all;
        return before;
    };
    for (int c = tid; c < lv.count; c += 1024) cid[lv.rank1[c / lv.per] * lv.per + lv.rank2[c]] = c;
    for (int l = tid; l <= lv.count; l += 1024) pos[l] = lv.off[(int64_t)l * lv.stride];
    __syncthreads();
    int cut[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int l = 2 * tid + h;
        cut[h] = 0;
        if (l < lv.count && pos[l + 1] > pos[l]) {
            int p = l - 1;
            while (p >= 0 && pos[p + 1] == pos[p]) --p;   // the last leaf with rows
            cut[h] = 1;
            if (p >= 0) {
                const float *a = lv.cent + (int64_t)cid[l] * DP, *b = lv.cent + (int64_t)cid[p] * DP;
                float d = 0.f;
                for (int t = 0; t < DP; ++t) d = fmaf(a[t] - b[t], a[t] - b[t], d);
                cut[h] = d > 2.f * (lv.var[cid[l]] + lv.var[cid[p]]) ? 1 : 0;
            }
        }
    }
    int runs;
    int r = scan2(cut[0], cut[1], &runs);
    if (cut[0]) run_pos[r++] = pos[2 * tid];
    if (cut[1]) run_pos[r] = pos[2 * tid + 1];
    if (tid == 0) run_pos[runs] = (int)n;
    __syncthreads();
    int cnt[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int x = 2 * tid + h;
        cnt[h] = x < runs ? (run_pos[x + 1] - run_pos[x] + kR - 1) / kR : 0;
    }
    int total;
    const int at = scan2(cnt[0], cnt[1], &total);
    if (2 * tid < runs) run_tile[2 * tid] = at;
    if (2 * tid + 1 < runs) run_tile[2 * tid + 1] = at + cnt[0];
    if (tid == 0) *T = total;
    __syncthreads();
    for (int t = tid; t < total; t += 1024) {
        int lo = 0, hi = runs;   // run_tile[lo] <= t < run_tile[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (run_tile[mid] <= t) lo = mid;
            else hi = mid;
        }
        const int p = run_pos[lo] + (t - run_tile[lo]) * kR;
        tile_pos[t] = p;
        tile_rows[t] = min(kR, run_pos[lo + 1] - p);
    }
}

// Block per tile: the record, the original ids (INT_MAX past the tile's rows;
// |y|^2 = NaN there, which no comparison accepts), the bounding sphere
// (centre: the mean, transposed by tile; radius inflated for its rounding;
// largest |y|^2).  `tiles` = tiles_max.
__global__ void __launch_bounds__(256)
pack_kernel(const float *__restrict__ Y, const float *__restrict__ ny, int DP, const int32_t *__restrict__ perm,
            int64_t tiles, const int32_t *__restrict__ tile_pos, int32_t *__restrict__ tile_rows,
            const int32_t *__restrict__ T, float *__restrict__ rec, int32_t *__restrict__ ids,
            float *__restrict__ cenT, float *__restrict__ rad, float *__restrict__ nmax) {
    __shared__ float ys[64][kR + 1];
    __shared__ float cen[64];
    __shared__ float red[2][8];
    const int64_t t = blockIdx.x;
    const int last = *T;
    if (t > last || (t == last && (last & 1) == 0)) return;   // an empty tile completes an odd count
    const int tid = threadIdx.x, rows = t < last ? tile_rows[t] : 0;
    const int64_t r0 = t < last ? tile_pos[t] : 0;
    if (t == last && tid == 0) tile_rows[t] = 0;
    // four lanes per row, 16-byte loads
    const int r = tid >> 2, l = tid & 3;
    const int64_t o = r < rows ? (int64_t)perm[r0 + r] : 0;
    float nn = 0.f;
    for (int c = l; c < DP / 4; c += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) v = reinterpret_cast<const float4 *>(Y + o * DP)[c];
        ys[4 * c][r] = v.x;
        ys[4 * c + 1][r] = v.y;
        ys[4 * c + 2][r] = v.z;
        ys[4 * c + 3][r] = v.w;
        nn = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, nn))));
    }
    nn += __shfl_xor_sync(0xffffffffu, nn, 1);
    nn += __shfl_xor_sync(0xffffffffu, nn, 2);
    if (l == 0) ids[t * kR + r] = r < rows ? (int32_t)o : INT_MAX;
    __syncthreads();
    float *out = rec + t * record_floats(DP);
    for (int e = tid; e < DP * kR; e += 256) out[e] = ys[e >> 6][e & 63];
    if (tid < kR) out[DP * kR + tid] = tid < rows ? ny[perm[r0 + tid]] : NAN;
    if (tid < DP) {
        float c = 0.f;
        for (int i = 0; i < rows; ++i) c += ys[tid][i];
        cen[tid] = rows > 0 ? c / (float)rows : 0.f;
        cenT[(int64_t)tid * tiles + t] = cen[tid];
    }
    __syncthreads();
    float dd = 0.f;
    if (r < rows)
        for (int c = l; c < DP; c += 4) {
            const float e = ys[c][r] - cen[c];
            dd = fmaf(e, e, dd);
        }
    dd += __shfl_xor_sync(0xffffffffu, dd, 1);
    dd += __shfl_xor_sync(0xffffffffu, dd, 2);
    // NaN must survive the maximum: a tile that holds one is never dropped
    const bool bad = !(dd < INFINITY) || !(nn < INFINITY);
    float md = bad ? INFINITY : dd, mn = r < rows ? nn : 0.f;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, s));
        mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, s));
    }
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = md;
        red[1][tid >> 5] = mn;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < 8; ++w) {
            md = fmaxf(md, red[0][w]);
            mn = fmaxf(mn, red[1][w]);
        }
        rad[t] = rows > 0 ? sqrtf(md) * (1.f + 0x1p-10f) + 1e-6f : -1.f;   // -1: an empty tile
        nmax[t] = mn;
    }
}

// --------------------------------------------------------------------- top-k

// The KC smallest s of one query in registers (RowTopK), fed through a
// per-thread shared-memory buffer as BufferedTopK is, with the row's bound as
// the filter.  Equal values beyond the list's end are dropped whatever their
// ids: such a row is finished by ties_kernel.
template <int KC>
struct List {
    RowTopK<KC> top;
    float bound;          // values above it cannot be among the k nearest
    float vv, v2;         // |y_i|^2 and |y_i|
    uint32_t sbase;
    int cnt, k, w;

    __device__ __forceinline__ void start(float nn, int k_, int w_) {
        top.init();
#pragma unroll
        for (int c = 0; c < KC; ++c) top.key[c] = FLT_MAX;   // finite: infinite values are never accepted
        bound = FLT_MAX;
        vv = nn;
        v2 = sqrtf(nn);
        cnt = 0;
        k = k_;
        w = w_;
    }
    __device__ __forceinline__ float reach_of(float t) const { return rr::reach(t, vv, v2, w); }
    __device__ __forceinline__ float reach() const {
        float t = top.key[0];
#pragma unroll
        for (int c = 1; c < KC; ++c) t = fmaxf(t, c < k ? top.key[c] : -FLT_MAX);   // ascending: the k-th
        return reach_of(t);
    }
    __device__ __forceinline__ void flush() {   // warp-synchronous
        const int rounds = __reduce_max_sync(0xffffffffu, cnt);
#pragma unroll 1
        for (int e = 0; e < rounds; ++e) {
            if (e < cnt) {
                float v;
                int j;
                const uint32_t a = sbase + (uint32_t)e * (4u * kQ);
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(j) : "r"(a + 4u * kQ * kCap) : "memory");
                if (v < top.thr()) top.insert(v, j);
            }
        }
        cnt = 0;
        bound = fminf(bound, fminf(top.thr(), reach()));
    }
    // An empty list whose first tile is known: the largest of its 16 minima
    // of four (k <= 16) or 32 minima of two bounds the k-th smallest, so what
    // lies beyond its reach never enters.  Any value that is no number leaves
    // it unbounded.
    __device__ __forceinline__ void start_bound(const float *row) {
        float most = -FLT_MAX;
        bool all = true;
#pragma unroll 4
        for (int c = 0; c < kR; c += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(row + c);
            const float a = fminf(v.x, v.y), b = fminf(v.z, v.w);
            most = fmaxf(most, k <= 16 ? fminf(a, b) : fmaxf(a, b));
            all = all && a < INFINITY && b < INFINITY;
        }
        if (all) bound = fminf(FLT_MAX, reach_of(most));
    }
    // Eight values of positions j0 .. j0 + 7 (warp-synchronous).  Eight at a
    // time and not sixteen: the buffer then fills to 13 of its 20 entries
    // before a flush, so the lanes' insertions share more of their rounds.
    __device__ __forceinline__ void offer8(const float (&v)[8], int j0) {
        const float lo = min8(v);
        const bool hit = lo <= bound;
        if (!__any_sync(0xffffffffu, hit)) return;
        if (__any_sync(0xffffffffu, hit && cnt > kCap - 8)) flush();
        const float t = bound;
        if (!(lo <= t)) return;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (v[i] <= t) {
                const uint32_t a = sbase + (uint32_t)cnt * (4u * kQ);
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v[i]) : "memory");
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(a + 4u * kQ * kCap), "r"(j0 + i) : "memory");
                ++cnt;
            }
        }
    }
};

__device__ __forceinline__ void fma2(uint64_t &d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t dup2(float x) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 split2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

struct Args {
    const float *rec;
    const int32_t *ids, *tile_pos, *tile_rows, *T;
    const float *cenT, *rad, *nmax;
    int64_t n, stride;      // rows; stride of cenT (tiles_max)
    int DP, width, k;
    float beta;
    int32_t *cand;          // [n, KC] positions, -1 for none
    int32_t *tie_rows;      // rows for ties_kernel
    float *tie_bound;       // (tie_rows: sorted position, then the row's place in the records)
    int *tie_count, *counter;
    uint32_t *bits;         // [CTAs][stride / 32] tiles an item keeps
    int32_t *big;           // [kBigItems][1 + kSeeds] items to be split, their seeds (-1 pads)
    int *big_count, *unit;  // their number (may exceed kBigItems), next part
    float *part_key;        // [query slots][part_segs][KC] lists of the parts; a slot is a query
    int32_t *part_id;       // tile pair's (split: position in `big`; flat: item) kQ rows
    int part_segs;
    float *vv;              // [query slots] |y|^2 (flat)
    unsigned long long *scanned;   // tiles scanned (a statistic)
    unsigned int *status;
    long long wait_budget;         // SM clocks a wait for a copy may take (tc_wait_budget)
};

// parts of a split item: segments of seg_tiles tiles
__device__ __forceinline__ int64_t seg_tiles(int64_t tiles) {
    const int64_t s = min((int64_t)kSegs, max((int64_t)1, tiles / kSegTiles));
    return ceil_div(tiles, s);
}

// The candidates of an item's query row, and the row itself for ties_kernel if
// more rows may lie within reach than the list holds.
template <int KC>
__device__ __forceinline__ void emit(const Args &g, const List<KC> &tk, int64_t item, int tid) {
    const int64_t q = g.tile_pos[2 * item + (tid >> 6)] + (tid & 63);
    int32_t *out = g.cand + q * KC;
    const float reach = tk.reach();
#pragma unroll
    for (int c = 0; c < KC; ++c) {
        out[c] = tk.top.key[c] <= reach ? tk.top.id[c] : -1;   // -1 also where empty
    }
    if (tk.top.id[KC - 1] >= 0 && tk.top.key[KC - 1] <= reach) {
        const int x = atomicAdd(g.tie_count, 1);
        g.tie_rows[2 * x] = (int32_t)q;
        g.tie_rows[2 * x + 1] = (int32_t)(item * kQ + tid);
        g.tie_bound[x] = reach;
    }
}

// kSplit = false: an item per query tile pair.  An item that keeps more than
// 1 / 16 of the tiles (a tile that holds a row far from its cluster, or spans
// two) would outlast all others on its CTA (100k rows: 10 ms for one); such
// items are put on a list instead, as long as it has room, and kSplit = true
// runs them in up to kSegs parts, each over a segment of the database from
// the item's own surroundings on, whose lists merge_kernel joins.
// kFlat: rows in their own order, part_segs parts per item and no tests: the
// search of fewer rows than an ordering pays for (see launch_knn_simt_flat).
enum { kWhole, kSplitItems, kFlat };
template <int KC, int kMode>
__global__ void __launch_bounds__(kQ, 2) simt_pruned_kernel(const Args g) {
    constexpr bool kSplit = kMode == kSplitItems, kIsFlat = kMode == kFlat;
    extern __shared__ __align__(128) uint8_t sm[];
    const int DP = g.DP;
    const Smem m = smem_layout(DP);
    float *xs = reinterpret_cast<float *>(sm + m.xs), *ys = reinterpret_cast<float *>(sm + m.ys);
    float *S = reinterpret_cast<float *>(sm + m.s);
    int *list = reinterpret_cast<int *>(sm + m.list);   // [kChunk]
    float *cen = reinterpret_cast<float *>(sm + m.cen);
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + m.bars);   // [kStages]
    uint64_t *xfull = full + kStages;
    volatile int *item_s = reinterpret_cast<volatile int *>(xfull + 1);
    float *redf = reinterpret_cast<float *>(const_cast<int *>(item_s) + 1);   // [4]
    uint32_t *masks = reinterpret_cast<uint32_t *>(redf + 4);                 // [kWords]
    int *seeds = reinterpret_cast<int *>(masks + kWords);                     // [kSeeds]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, qg = tid >> 3, rg = tid & 7;
    const int rf = record_floats(DP);
    const uint32_t rec_bytes = (uint32_t)rf * 4u, x_bytes = (uint32_t)DP * kR * 4u;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) tc::mbar_init(&full[s], 1);
        tc::mbar_init(xfull, 1);
        tc::fence_barrier_init();
    }
    __syncthreads();
    List<KC> tk;
    tk.sbase = (uint32_t)__cvta_generic_to_shared(reinterpret_cast<float *>(sm + m.buf) + tid);
    // bounded; a budget shorter than a few sleeps is polled
    const uint32_t sleep_ns = g.wait_budget < 8 * (long long)kSleepNs ? 0 : kSleepNs;
    auto wait = [&](uint64_t *bar, uint32_t parity, long long budget) -> bool {
        if (tc::mbar_arrived(bar, parity, sleep_ns)) return true;
        const long long t0 = clock64();
        while (!tc::mbar_arrived(bar, parity, sleep_ns))
            if (clock64() - t0 > budget) {
                record_status(g.status, RSC_ERR_TIMEOUT);
                return false;
            }
        return true;
    };
    const int64_t tiles = *g.T;   // an odd count is followed by an empty tile
    const int64_t seg_len = kIsFlat ? ceil_div(tiles, (int64_t)g.part_segs) : seg_tiles(tiles);
    const int segs = kIsFlat ? g.part_segs : (int)ceil_div(tiles, seg_len);
    const int64_t pairs = ceil_div(tiles, (int64_t)2);
    const int64_t units = kIsFlat ? pairs * segs : kSplit ? (int64_t)min(*g.big_count, kBigItems) * segs : pairs;
    uint32_t tile_no = 0;     // tiles consumed by this CTA so far (stage tile_no % kStages)
    uint32_t items = 0;
    unsigned long long scanned = 0;
    auto issue = [&](uint32_t no, int64_t t) {   // thread 0: the copies of tile t as the CTA's tile number `no`
        const int s = no % kStages;
        tc::mbar_arrive_expect_tx(&full[s], rec_bytes);
        tc::bulk_load(ys + s * rf, g.rec + t * rf, rec_bytes, &full[s]);
    };
    // scans tiles list[0 .. nl); false when a copy did not arrive (the
    // whole CTA then leaves, after the copies in flight have had their time)
    auto scan = [&](int nl, bool first) -> bool {
        if (tid == 0) {
            issue(tile_no, list[0]);
            if (nl > 1) issue(tile_no + 1, list[1]);
        }
        for (int i = 0; i < nl; ++i, ++tile_no) {
            const int s = tile_no % kStages;
            const bool ok = wait(&full[s], (tile_no / kStages) & 1, g.wait_budget);
            uint64_t acc[8][4];
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = 0ull;
            const float *yb = ys + s * rf;
            auto step = [&](int t) {
                const float4 xa = *reinterpret_cast<const float4 *>(xs + t * kR + 4 * qg);
                const float4 xb = *reinterpret_cast<const float4 *>(xs + (DP + t) * kR + 4 * qg);
                const ulonglong2 y0 = *reinterpret_cast<const ulonglong2 *>(yb + t * kR + 4 * rg);
                const ulonglong2 y1 = *reinterpret_cast<const ulonglong2 *>(yb + t * kR + 32 + 4 * rg);
                const uint64_t yv[4] = {y0.x, y0.y, y1.x, y1.y};
                const float xv[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const uint64_t x2 = dup2(xv[a]);
#pragma unroll
                    for (int b = 0; b < 4; ++b) fma2(acc[a][b], x2, yv[b]);
                }
            };
            // four components per trip; those at `width` and beyond are zero
            // and are skipped (an FMA of two zeros leaves s unchanged)
            int t = 0;
#pragma unroll 1
            for (; t + 4 <= g.width; t += 4) {
#pragma unroll
                for (int u = 0; u < 4; ++u) step(t + u);
            }
#pragma unroll 1
            for (; t < g.width; ++t) step(t);
            // every read of the previous s tile is done
            if (__syncthreads_or(!ok)) {
                if (tid == 0) {   // the copies in flight get their time again
                    wait(&full[s], (tile_no / kStages) & 1, kDrainBudget);
                    if (i + 1 < nl) wait(&full[(tile_no + 1) % kStages], ((tile_no + 1) / kStages) & 1, kDrainBudget);
                }
                return false;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 nv = *reinterpret_cast<const float4 *>(yb + DP * kR + 32 * h + 4 * rg);
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const float2 p = split2(acc[a][2 * h]), q = split2(acc[a][2 * h + 1]);
                    float *row = S + (a < 4 ? 4 * qg + a : 64 + 4 * qg + a - 4) * kPitch;
                    *reinterpret_cast<float4 *>(row + 32 * h + 4 * rg) =
                        make_float4(fmaf(-2.f, p.x, nv.x), fmaf(-2.f, p.y, nv.y), fmaf(-2.f, q.x, nv.z),
                                    fmaf(-2.f, q.y, nv.w));
                }
            }
            __syncthreads();   // the s tile is in place; the stage is free
            if (tid == 0 && i + 2 < nl) issue(tile_no + 2, list[i + 2]);
            const float *sr = S + tid * kPitch;
            const int tt = list[i], j0 = g.tile_pos[tt];
            if (first && i == 0 && g.tile_rows[tt] == kR) tk.start_bound(sr);   // a full tile, empty lists
#pragma unroll 1
            for (int h = 0; h < kR; h += 8) {
                const float4 lo = *reinterpret_cast<const float4 *>(sr + h), hi = *reinterpret_cast<const float4 *>(sr + h + 4);
                const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                tk.offer8(v, j0 + h);
            }
        }
        scanned += nl;
        tk.flush();
        __syncthreads();   // the list may be rewritten
        return true;
    };
    for (;; ++items) {
        __syncthreads();
        if (tid == 0) *item_s = atomicAdd(kSplit ? g.unit : g.counter, 1);
        __syncthreads();
        const int64_t unit = *item_s;
        if (unit >= units) break;
        const int32_t *big = g.big + unit / segs * (1 + kSeeds);   // kSplit
        const int64_t item = kSplit ? (int64_t)big[0] : kIsFlat ? unit / segs : unit;
        if (tid == 0) {
            tc::mbar_arrive_expect_tx(xfull, 2 * x_bytes);
            tc::bulk_load(xs, g.rec + (2 * item) * rf, x_bytes, xfull);
            tc::bulk_load(xs + DP * kR, g.rec + (2 * item + 1) * rf, x_bytes, xfull);
        }
        // centres of the two query tiles
        if (!kIsFlat) {
            const int h = tid >> 6, u = tid & 63;
            cen[tid] = u < DP ? g.cenT[(int64_t)u * g.stride + 2 * item + h] : 0.f;
        }
        const bool got = wait(xfull, items & 1, g.wait_budget);
        if (__syncthreads_or(!got)) {
            if (tid == 0) wait(xfull, items & 1, kDrainBudget);
            return;
        }
        const bool live = (tid & 63) < g.tile_rows[2 * item + (tid >> 6)];
        float nn = 0.f;
        const float *xr = xs + (tid >> 6) * DP * kR + (tid & 63);
        for (int t = 0; t < g.width; ++t) nn = fmaf(xr[t * kR], xr[t * kR], nn);
        tk.start(nn, g.k, g.width);
        float rq[2] = {0.f, 0.f}, nq[2] = {0.f, 0.f};
        if (!kIsFlat) {
            rq[0] = g.rad[2 * item];
            rq[1] = g.rad[2 * item + 1];
            nq[0] = g.nmax[2 * item];
            nq[1] = g.nmax[2 * item + 1];
        }
        const int wlo = (int)max((int64_t)0, 2 * item - kWin), whi = (int)min(tiles, 2 * item + 2 + kWin);
        // the range of tiles in chunks, from the chunk of the query tiles on
        const int64_t lo = kMode != kWhole ? min(tiles, (unit % segs) * seg_len) : 0;
        const int64_t hi = kMode != kWhole ? min(tiles, lo + seg_len) : tiles;
        const int chunks = (int)ceil_div(hi - lo, (int64_t)kChunk), c0 = kSplit ? 0 : (int)((2 * item) / kChunk);
        const int64_t most = max((int64_t)64, tiles / 16);
        uint32_t *bits = g.bits + (int64_t)blockIdx.x * ceil_div(tiles, (int64_t)kChunk) * kWords;
        // The lists live in registers, so there is one scan call, and what it
        // scans next is worked out in steps:
        //   kWindow  the tiles around the query tiles
        //   kMark    (no scan) which tiles the bounds keep then, and the
        //            nearest tiles; few kept tiles: on to kChunks
        //   kNearest many: the window did not bound the rows (an ordering that
        //            put them beside strangers); the nearest tiles first
        //   kAgain   (no scan) the marks once more; still many: the item is split
        //   kChunks  the marked tiles, chunk by chunk, tested against the
        //            bounds as they are by then
        // A part of a split item goes from kWindow over its seeds to kChunks.
        enum { kWindow, kMark, kNearest, kAgain, kChunks };
        int step = kWindow, ci = 0, n_seeds = 0;
        int64_t kept = 0;
        float near_d[2] = {INFINITY, INFINITY}, tq[2] = {INFINITY, INFINITY};
        int near_t[2] = {-1, -1};
        bool fresh = true, deferred = false;   // fresh: tq must be taken anew
        if (kSplit) {
            if (tid < kSeeds) seeds[tid] = big[1 + tid];
            while (n_seeds < kSeeds && big[1 + n_seeds] >= 0) ++n_seeds;
        }
        int64_t done = 0;   // flat: tiles of the part scanned so far
        bool first = true;
        while (true) {
            int nl = 0;
            if (kIsFlat) {   // the part's tiles, from the query's own on when they are among them
                const int64_t len = hi - lo, from = 2 * item >= lo && 2 * item < hi ? 2 * item - lo : 0;
                nl = (int)min((int64_t)kChunk, len - done);
                if (nl <= 0) break;
                for (int x = tid; x < nl; x += kQ) {
                    const int64_t at = from + done + x;
                    list[x] = (int)(lo + (at < len ? at : at - len));
                }
                done += nl;
            } else if (step == kWindow) {
                nl = whi - wlo;
                const int own = (int)(2 * item) - wlo;   // the query tiles themselves first
                if (tid < nl) list[tid] = wlo + (tid == 0 ? own : tid <= own ? tid - 1 : tid);
            } else if (step == kNearest) {
                nl = n_seeds;
                if (tid < nl) list[tid] = seeds[tid];
            } else {
                if (ci == chunks) {
                    if (step == kChunks) break;
                    ci = 0;
                    if (kept > most && step == kMark) {   // the nearest tile of every (warp, half)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
#pragma unroll
                            for (int o = 16; o > 0; o >>= 1) {
                                const float od = __shfl_xor_sync(0xffffffffu, near_d[h], o);
                                const int ot = __shfl_xor_sync(0xffffffffu, near_t[h], o);
                                if (od < near_d[h] || (od == near_d[h] && ot < near_t[h])) {
                                    near_d[h] = od;
                                    near_t[h] = ot;
                                }
                            }
                            if (lane == 0) masks[2 * warp + h] = (uint32_t)near_t[h];
                        }
                        __syncthreads();
                        if (tid == 0) {
                            int m = 0;
                            for (int x = 0; x < kSeeds; ++x) {
                                const int t = (int)masks[x];
                                bool have = t < 0;
                                for (int y = 0; y < m; ++y) have |= seeds[y] == t;
                                if (!have) seeds[m++] = t;
                            }
                            *item_s = m;
                            for (; m < kSeeds; ++m) seeds[m] = -1;
                        }
                        __syncthreads();
                        n_seeds = *item_s;
                        step = kNearest;
                        continue;
                    }
                    if (kept > most && step == kAgain) {
                        if (tid == 0) {
                            const int at = atomicAdd(g.big_count, 1);
                            *item_s = at < kBigItems;
                            if (at < kBigItems) {
                                g.big[at * (1 + kSeeds)] = (int32_t)item;
                                for (int x = 0; x < kSeeds; ++x) g.big[at * (1 + kSeeds) + 1 + x] = seeds[x];
                            }
                        }
                        __syncthreads();
                        deferred = *item_s != 0;
                        if (deferred) break;
                    }
                    step = kChunks;
                    continue;
                }
                const int chunk = c0 + ci < chunks ? c0 + ci : c0 + ci - chunks;
                const int64_t base = lo + (int64_t)chunk * kChunk;
                uint32_t *word = bits + chunk * kWords;
                ++ci;
                const bool all = kSplit || step == kMark;
                if (!all) {
                    uint32_t any = 0;
#pragma unroll
                    for (int x = 0; x < kWords; ++x) any |= word[x];
                    if (any == 0) continue;
                }
                if (fresh) {   // the tiles' bounds (dead rows ask for nothing)
                    float tau = live ? tk.bound + tk.vv : -INFINITY;
                    if (live && !(tau < INFINITY)) tau = INFINITY;   // also NaN
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) tau = fmaxf(tau, __shfl_xor_sync(0xffffffffu, tau, o));
                    if (lane == 0) redf[warp] = tau;
                    __syncthreads();
                    tq[0] = fmaxf(redf[0], redf[1]);
                    tq[1] = fmaxf(redf[2], redf[3]);
                    fresh = false;
                }
#pragma unroll 1
                for (int j = 0; j < kChunk / kQ; ++j) {
                    const int x = j * kQ + tid;
                    const int64_t t = base + x;
                    bool keep = false;
                    if (all ? t < hi && (t < wlo || t >= whi) : (word[x >> 5] >> lane & 1u) != 0) {
                        const float rt = g.rad[t], nt = g.nmax[t];
                        float a[2] = {0.f, 0.f};
#pragma unroll 8
                        for (int u = 0; u < g.width; ++u) {
                            const float c = g.cenT[(int64_t)u * g.stride + t];
                            const float e0 = cen[u] - c, e1 = cen[64 + u] - c;
                            a[0] = fmaf(e0, e0, a[0]);
                            a[1] = fmaf(e1, e1, a[1]);
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float gap = sqrtf(a[h]) - rq[h] - rt;
                            const bool drop = gap > 0.f && gap * gap - g.beta * nt - 0x1p-11f * (nq[h] + nt) > tq[h];
                            keep |= rq[h] >= 0.f && !drop;   // -1: an empty tile
                            if (rq[h] >= 0.f && a[h] < near_d[h]) {
                                near_d[h] = a[h];
                                near_t[h] = (int)t;
                            }
                        }
                        if (step != kMark)
                            for (int y = 0; y < n_seeds; ++y) keep &= seeds[y] != (int)t;
                    }
                    const unsigned b = __ballot_sync(0xffffffffu, keep);
                    if (lane == 0) masks[x >> 5] = b;
                }
                __syncthreads();
                if (step == kChunks) {
#pragma unroll
                    for (int wd = 0; wd < kWords; ++wd) {
                        const uint32_t b = masks[wd];
                        if (wd % 4 == warp && (b >> lane & 1u))
                            list[nl + __popc(b & ((1u << lane) - 1u))] = (int)base + wd * 32 + lane;
                        nl += __popc(b);
                    }
                } else {
                    if (tid < kWords) word[tid] = masks[tid];
#pragma unroll
                    for (int wd = 0; wd < kWords; ++wd) kept += __popc(masks[wd]);
                }
            }
            __syncthreads();
            if (nl > 0) {
                if (!scan(nl, first)) return;
                fresh = true;
                first = false;
            }
            if (kIsFlat) continue;
            if (step == kWindow) step = kSplit ? (n_seeds > 0 ? kNearest : kChunks) : kMark;
            else if (step == kNearest) {
                step = kSplit ? kChunks : kAgain;
                kept = 0;
            }
        }
        if (kMode != kWhole) {
            const int64_t slot = (kIsFlat ? item : unit / segs) * kQ + tid;
            if (live) {
                float *pk = g.part_key + (slot * g.part_segs + unit % segs) * KC;
                int32_t *pi = g.part_id + (slot * g.part_segs + unit % segs) * KC;
#pragma unroll
                for (int c = 0; c < KC; c += 4) {
                    *reinterpret_cast<float4 *>(pk + c) =
                        make_float4(tk.top.key[c], tk.top.key[c + 1], tk.top.key[c + 2], tk.top.key[c + 3]);
                    *reinterpret_cast<int4 *>(pi + c) =
                        make_int4(tk.top.id[c], tk.top.id[c + 1], tk.top.id[c + 2], tk.top.id[c + 3]);
                }
                if (kIsFlat && unit % segs == 0) g.vv[slot] = nn;
            }
        } else if (live && !deferred) {
            emit(g, tk, item, tid);
        }
    }
    if (tid == 0 && scanned) atomicAdd(g.scanned, scanned);
}

// Joins the lists of a split item's parts (every part scanned the tiles around
// the query tiles, so those entries come more than once).
template <int KC>
__global__ void __launch_bounds__(kQ) merge_kernel(const Args g) {
    const int64_t tiles = *g.T;
    const int segs = (int)ceil_div(tiles, seg_tiles(tiles));
    const int b = blockIdx.x, tid = threadIdx.x;
    if (b >= min(*g.big_count, kBigItems)) return;
    const int64_t item = g.big[b * (1 + kSeeds)];
    if ((tid & 63) >= g.tile_rows[2 * item + (tid >> 6)]) return;
    const float *xr = g.rec + (2 * item + (tid >> 6)) * record_floats(g.DP) + (tid & 63);
    float nn = 0.f;
    for (int t = 0; t < g.width; ++t) nn = fmaf(xr[t * kR], xr[t * kR], nn);
    List<KC> tk;
    tk.start(nn, g.k, g.width);
    for (int s = 0; s < segs; ++s) {
        const int64_t at = (((int64_t)b * kQ + tid) * g.part_segs + s) * KC;
#pragma unroll 1
        for (int c = 0; c < KC; ++c) {
            const float v = g.part_key[at + c];
            const int j = g.part_id[at + c];
            if (j < 0 || !(v < tk.top.thr())) break;   // ascending
            bool have = false;
#pragma unroll
            for (int x = 0; x < KC; ++x) have |= tk.top.id[x] == j;
            if (!have) tk.top.insert(v, j);
        }
    }
    emit(g, tk, item, tid);
}

// Rows whose list was too short for the rows within reach: a warp scans every
// tile (lane per database row, the same FMA chain for s), scores the rows at
// or below the bound with the re-rank's arithmetic and keeps the k <= 32
// smallest (distance, id), one per lane.  Integer-like data with more equal
// distances than a list holds come here; others hardly ever do.
__global__ void __launch_bounds__(128)
ties_kernel(const Args g, const float *__restrict__ R, int64_t rs, int d, bool cosine, bool vec,
            int32_t *__restrict__ idx, float *__restrict__ dist) {
    __shared__ float xs[4][64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int count = *g.tie_count;
    const int rf = record_floats(g.DP);
    for (int64_t x = (int64_t)blockIdx.x * 4 + warp; x < count; x += (int64_t)gridDim.x * 4) {
        const int64_t q = g.tie_rows[2 * x], slot = g.tie_rows[2 * x + 1];
        const float bound = g.tie_bound[x];
        const float *xr = g.rec + (slot / kR) * rf + slot % kR;
        __syncwarp();
        for (int t = lane; t < g.width; t += 32) xs[warp][t] = xr[(int64_t)t * kR];
        __syncwarp();
        float qv[8];
        rr::load8(R + q * rs, lane & 7, d, cosine, vec, qv);
        const bool fq = cosine && R[q * rs + d] != 0.f;
        float bk = INFINITY;   // lane's entry of the sorted list
        int bi = INT_MAX;
        const int64_t slots = (int64_t)*g.T * kR;
        for (int64_t j0 = 0; j0 < slots; j0 += 32) {
            const float *yr = g.rec + (j0 / kR) * rf + (j0 % kR) + lane;
            float acc = 0.f;
            for (int t = 0; t < g.width; ++t) acc = fmaf(xs[warp][t], yr[t * kR], acc);
            const float s = fmaf(-2.f, acc, yr[g.DP * kR]);
            unsigned hits = __ballot_sync(0xffffffffu, s <= bound);
            while (hits) {
                const int64_t sj = j0 + __ffs(hits) - 1;   // place in the records
                const int64_t j = g.tile_pos[sj / kR] + sj % kR;
                hits &= hits - 1;
                float yv[8];
                rr::load8(R + j * rs, lane & 7, d, cosine, vec, yv);
                float key = rr::dist2(qv, yv);
                if (cosine) {
                    const bool fy = R[j * rs + d] != 0.f;
                    if (fq || fy) key = (fq && fy) ? 0.f : 2.f;
                }
                const int id = g.ids[sj];
                const bool less = bk < key || (bk == key && bi < id);   // this lane's entry stays before it
                const int at = __popc(__ballot_sync(0xffffffffu, less));
                const float pk = __shfl_up_sync(0xffffffffu, bk, 1);
                const int pi = __shfl_up_sync(0xffffffffu, bi, 1);
                if (lane == at) {
                    bk = key;
                    bi = id;
                } else if (lane > at) {
                    bk = pk;
                    bi = pi;
                }
            }
        }
        const int64_t o = g.ids[slot];
        if (lane < g.k) {
            idx[o * g.k + lane] = bi != INT_MAX ? bi : -1;
            dist[o * g.k + lane] = bi != INT_MAX ? (cosine ? 0.5f * bk : sqrtf(bk)) : INFINITY;
        }
    }
}

constexpr int kCounters = 7;
constexpr int kMaxList = 40;

struct Layout {
    float *rec, *cenT, *rad, *nmax, *tie_bound;
    int32_t *ids, *tile_pos, *tile_rows, *tie_rows;
    int *counters;   // tie_count, counter, scanned (64 bits), tiles, big_count, unit
    int32_t *big, *part_id;
    uint32_t *bits;
    float *part_key;
    size_t bytes;
};
Layout layout(void *scratch, int64_t n, int DP) {
    Carve cv(scratch);
    Layout L;
    const int64_t tiles = tiles_max(n);
    L.rec = cv.take<float>((size_t)tiles * record_floats(DP));
    L.ids = cv.take<int32_t>((size_t)tiles * kR);
    L.cenT = cv.take<float>((size_t)tiles * DP);
    L.rad = cv.take<float>((size_t)tiles);
    L.nmax = cv.take<float>((size_t)tiles);
    L.tile_pos = cv.take<int32_t>((size_t)tiles);
    L.tile_rows = cv.take<int32_t>((size_t)tiles);
    L.tie_rows = cv.take<int32_t>((size_t)2 * n);
    L.tie_bound = cv.take<float>((size_t)n);
    L.counters = cv.take<int>(kCounters);
    L.big = cv.take<int32_t>(kBigItems * (1 + kSeeds));
    L.bits = cv.take<uint32_t>((size_t)kMaxCtas * ceil_div(tiles, (int64_t)kChunk) * kWords);
    const size_t parts = (size_t)kBigItems * kSegs * kMaxList * kQ;
    L.part_key = cv.take<float>(parts);
    L.part_id = cv.take<int32_t>(parts);
    L.bytes = cv.used;
    return L;
}

Args make_args(const Layout &L, int64_t n, int DP, int width, int k, int metric, int32_t *cand, unsigned int *status) {
    Args g;
    g.rec = L.rec;
    g.ids = L.ids;
    g.cenT = L.cenT;
    g.rad = L.rad;
    g.nmax = L.nmax;
    g.tile_pos = L.tile_pos;
    g.tile_rows = L.tile_rows;
    g.T = L.counters + 4;
    g.n = n;
    g.stride = tiles_max(n);
    g.DP = DP;
    g.width = width;
    g.k = k;
    g.beta = metric == RSC_COSINE ? 1.f : 0.f;
    g.cand = cand;
    g.tie_rows = L.tie_rows;
    g.tie_bound = L.tie_bound;
    g.tie_count = L.counters;
    g.counter = L.counters + 1;
    g.scanned = reinterpret_cast<unsigned long long *>(L.counters + 2);
    g.bits = L.bits;
    g.big = L.big;
    g.big_count = L.counters + 5;
    g.unit = L.counters + 6;
    g.part_key = L.part_key;
    g.part_id = L.part_id;
    g.part_segs = kSegs;
    g.vv = nullptr;
    g.status = status;
    g.wait_budget = tc_wait_budget();
    return g;
}

}  // namespace simtp

// Entries beyond k: enough that rows within rounding of the k-th hardly ever
// fill the list.
int simt_pruned_list(int k) { return k <= 16 ? 24 : k <= 32 ? 40 : 0; }

size_t simt_pruned_scratch_bytes(int64_t n, int DP) { return simtp::layout(nullptr, n, DP).bytes; }

const unsigned long long *simt_pruned_scanned(void *scratch, int64_t n, int DP) {
    return reinterpret_cast<unsigned long long *>(simtp::layout(scratch, n, DP).counters + 2);
}

namespace simtp {

template <int KC>
cudaError_t launch_list(const Args &g, int64_t tiles, cudaStream_t st) {
    const int smem = smem_layout(g.DP).total;
    auto whole = simt_pruned_kernel<KC, kWhole>;
    auto split = simt_pruned_kernel<KC, kSplitItems>;
    cudaError_t e = cudaFuncSetAttribute(whole, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(split, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    whole<<<(unsigned)std::min<int64_t>(tiles / 2, std::min(kMaxCtas, 2 * sm_count())), kQ, smem, st>>>(g);
    split<<<(unsigned)std::min<int64_t>(kBigItems * kSegs, 2 * sm_count()), kQ, smem, st>>>(g);
    merge_kernel<KC><<<kBigItems, kQ, 0, st>>>(g);
    return cudaGetLastError();
}

}  // namespace simtp

OrderTarget simt_pruned_target() { return {128, true}; }

cudaError_t launch_knn_simt_pruned(const float *Y, const float *ny, int64_t n, int DP, int width, int k, int metric,
                                   const int32_t *perm, const OrderLeaves &leaves, void *scratch, int32_t *cand,
                                   unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    const Layout L = layout(scratch, n, DP);
    const int64_t tiles = tiles_max(n);
    cudaError_t e = cudaMemsetAsync(L.counters, 0, kCounters * sizeof(int), st);
    if (e != cudaSuccess) return e;
    tile_table_kernel<<<1, 1024, 0, st>>>(leaves, n, DP, L.tile_pos, L.tile_rows, L.counters + 4);
    pack_kernel<<<(unsigned)tiles, 256, 0, st>>>(Y, ny, DP, perm, tiles, L.tile_pos, L.tile_rows, L.counters + 4, L.rec,
                                                 L.ids, L.cenT, L.rad, L.nmax);
    const Args g = make_args(L, n, DP, width, k, metric, cand, status);
    return simt_pruned_list(k) == 24 ? launch_list<24>(g, tiles, st) : launch_list<kMaxList>(g, tiles, st);
}

cudaError_t launch_simt_ties(int64_t n, int d, int DP, int width, int k, int metric, void *scratch, const float *R,
                             int64_t rs, int32_t *idx, float *dist, cudaStream_t st) {
    using namespace simtp;
    const Layout L = layout(scratch, n, DP);
    const Args g = make_args(L, n, DP, width, k, metric, nullptr, nullptr);
    const bool vec = rs % 4 == 0 && reinterpret_cast<uintptr_t>(R) % 16 == 0;
    ties_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n, (int64_t)4), 8 * sm_count()), 128, 0, st>>>(
        g, R, rs, d, metric == RSC_COSINE, vec, idx, dist);
    return cudaGetLastError();
}

// ------------------------------------------------------------- rows as they are

namespace simtp {

// Block per tile of 64 rows in their own order: record, ids, tile tables (the
// tile that completes an odd count is empty).
__global__ void __launch_bounds__(256)
pack_flat_kernel(const float *__restrict__ Y, const float *__restrict__ ny, int64_t n, int DP, float *__restrict__ rec,
                 int32_t *__restrict__ ids, int32_t *__restrict__ tile_pos, int32_t *__restrict__ tile_rows,
                 int32_t *__restrict__ T) {
    __shared__ float ys[64][kR + 1];
    const int64_t t = blockIdx.x, r0 = t * kR;
    const int tid = threadIdx.x, rows = (int)max((int64_t)0, min((int64_t)kR, n - r0));
    const int r = tid >> 2, l = tid & 3;
    for (int c = l; c < DP / 4; c += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) v = reinterpret_cast<const float4 *>(Y + (r0 + r) * DP)[c];
        ys[4 * c][r] = v.x;
        ys[4 * c + 1][r] = v.y;
        ys[4 * c + 2][r] = v.z;
        ys[4 * c + 3][r] = v.w;
    }
    if (l == 0) ids[r0 + r] = r < rows ? (int32_t)(r0 + r) : INT_MAX;
    __syncthreads();
    float *out = rec + t * record_floats(DP);
    for (int e = tid; e < DP * kR; e += 256) out[e] = ys[e >> 6][e & 63];
    if (tid < kR) out[DP * kR + tid] = tid < rows ? ny[r0 + tid] : NAN;
    if (tid == 0) {
        tile_pos[t] = (int32_t)r0;
        tile_rows[t] = rows;
        if (t == 0) *T = (int32_t)ceil_div(n, (int64_t)kR);
    }
}

struct FlatLayout {
    float *rec, *part_key, *vv, *tie_bound;
    int32_t *ids, *tile_pos, *tile_rows, *part_id, *tie_rows;
    int *counters;   // tie_count, counter, scanned (64 bits), tiles
    size_t bytes;
};
FlatLayout flat_layout(void *scratch, int64_t n, int DP, int k) {
    Carve cv(scratch);
    FlatLayout L;
    const int64_t items = ceil_div(n, (int64_t)kQ);
    const size_t parts = (size_t)items * kQ * simt_flat_segs(n, DP) * simt_pruned_list(k);
    L.rec = cv.take<float>((size_t)items * 2 * record_floats(DP));
    L.ids = cv.take<int32_t>((size_t)items * kQ);
    L.tile_pos = cv.take<int32_t>((size_t)items * 2);
    L.tile_rows = cv.take<int32_t>((size_t)items * 2);
    L.part_key = cv.take<float>(parts);
    L.part_id = cv.take<int32_t>(parts);
    L.vv = cv.take<float>((size_t)items * kQ);
    L.tie_rows = cv.take<int32_t>((size_t)2 * n);
    L.tie_bound = cv.take<float>((size_t)n);
    L.counters = cv.take<int>(5);
    L.bytes = cv.used;
    return L;
}

Args flat_args(const FlatLayout &L, int64_t n, int DP, int width, int k, unsigned int *status) {
    Args g = {};
    g.rec = L.rec;
    g.ids = L.ids;
    g.tile_pos = L.tile_pos;
    g.tile_rows = L.tile_rows;
    g.tie_count = L.counters;
    g.counter = L.counters + 1;
    g.scanned = reinterpret_cast<unsigned long long *>(L.counters + 2);
    g.T = L.counters + 4;
    g.n = n;
    g.DP = DP;
    g.width = width;
    g.k = k;
    g.part_key = L.part_key;
    g.part_id = L.part_id;
    g.part_segs = simt_flat_segs(n, DP);
    g.vv = L.vv;
    g.tie_rows = L.tie_rows;
    g.tie_bound = L.tie_bound;
    g.status = status;
    g.wait_budget = tc_wait_budget();
    return g;
}

}  // namespace simtp

// Why parts and this kernel below kSimtPruneMinRows: the full scan's kernel
// keeps 32 values per row and split and its re-rank scores them all (10,000
// rows: 491 + 267 us, 2,700 rows: 105 + 120 us); here a list takes in only what
// can be among the k nearest and the re-rank scores what the merged lists leave
// (409 + 22 us and 61 + 12 us).
// Parts per query tile pair: the count whose waves of persistent CTAs cost
// least, a part costing its tiles plus about three (lists built anew, the
// query tiles fetched).
int simt_flat_segs(int64_t n, int DP) {
    const int64_t items = ceil_div(n, (int64_t)simtp::kQ), tiles = ceil_div(n, (int64_t)simtp::kR);
    const int64_t slots = 152 * (DP <= 56 ? 2 : 1);   // CTAs an SM holds
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int s = 1; s <= kSimtFlatSegs && s <= tiles; ++s) {
        const int64_t c = ceil_div(items * s, slots) * (ceil_div(tiles, (int64_t)s) + 3);
        if (c < cost) {
            cost = c;
            best = s;
        }
    }
    return best;
}

size_t simt_flat_scratch_bytes(int64_t n, int DP, int k) { return simtp::flat_layout(nullptr, n, DP, k).bytes; }

SimtParts simt_flat_parts(void *scratch, int64_t n, int DP, int k) {
    const simtp::FlatLayout L = simtp::flat_layout(scratch, n, DP, k);
    return {L.part_key, L.part_id, L.vv, simt_flat_segs(n, DP), simt_pruned_list(k), L.counters, L.tie_rows, L.tie_bound};
}

cudaError_t launch_knn_simt_flat(const float *Y, const float *ny, int64_t n, int DP, int width, int k, void *scratch,
                                 unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    const FlatLayout L = flat_layout(scratch, n, DP, k);
    const Args g = flat_args(L, n, DP, width, k, status);
    cudaError_t e = cudaMemsetAsync(L.counters, 0, 5 * sizeof(int), st);
    if (e != cudaSuccess) return e;
    const int64_t items = ceil_div(n, (int64_t)kQ);
    pack_flat_kernel<<<(unsigned)(2 * items), 256, 0, st>>>(Y, ny, n, DP, L.rec, L.ids, L.tile_pos, L.tile_rows,
                                                           L.counters + 4);
    const int smem = smem_layout(DP).total;
    auto kern = simt_pruned_list(k) == 24 ? simt_pruned_kernel<24, kFlat> : simt_pruned_kernel<kMaxList, kFlat>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
    kern<<<(unsigned)std::min<int64_t>(items * g.part_segs, 2 * sm_count()), kQ, smem, st>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_simt_flat_ties(int64_t n, int d, int DP, int width, int k, int metric, void *scratch, const float *R,
                                  int64_t rs, int32_t *idx, float *dist, cudaStream_t st) {
    using namespace simtp;
    const Args g = flat_args(flat_layout(scratch, n, DP, k), n, DP, width, k, nullptr);
    const bool vec = rs % 4 == 0 && reinterpret_cast<uintptr_t>(R) % 16 == 0;
    ties_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n, (int64_t)4), 8 * sm_count()), 128, 0, st>>>(
        g, R, rs, d, metric == RSC_COSINE, vec, idx, dist);
    return cudaGetLastError();
}

}  // namespace rsc
