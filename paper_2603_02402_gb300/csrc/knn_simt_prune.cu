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
// a second search of its item (kTies), which scores every row within the bound
// by the re-rank's own arithmetic.
//
// Tiles hold 64 consecutive rows, cut anew wherever two successive leaves of
// the ordering lie apart (the tile before is padded): a tile across such a gap
// spans two clusters, and its sphere keeps nearly every tile (100k rows, 60
// clusters, tiles cut every 64 rows whatever the leaves: 10.9 % of the pairs
// scanned and a few items that scanned everything, 15.4 ms).
//
// Persistent CTAs, two per SM; an item is two tiles of query rows, each with its own
// sphere and tau (the database tile is scanned when either keeps it).  The CTA
// scans the tiles around its own, then walks the database in chunks of 256 tiles
// from its own chunk on: tests every tile's sphere against its current taus, and
// scans the tiles that are left.  A tile's record (64 rows transposed, then
// |y|^2) is one contiguous block, brought in by a bulk copy two tiles ahead.
// A thread accumulates an 8 x 8 block of (query, row) pairs by packed FP32
// fused multiply-adds (fma.rn.f32x2: two pairs per instruction, each rounded
// as the scalar one; half the issue slots), then scans its own query's row of
// the s tile with the register top-k.
//
// What bounds it: the FMA pipe and, next to it, the insertions (a row takes in
// about 70 values).  50 components, k = 15, one GB300, whole call (in brackets
// the full scan): 100,003 rows, 60 clusters 1.58 ms (25.9), of which this kernel
// 0.8 and the ordering 0.5; 1M rows, 100 clusters 33 ms (2058).  Rows without any
// clusters, of which no tile is dropped (in the second brackets with every item
// run whole or, the first 192, in eight parts that each scanned the item's
// surroundings again): 1.58 ms (1.47) (1.69) at 16,384 rows, 1.99 (2.13) (2.41) at
// 20,000, 2.45 (2.72) (4.03) at 24,000, 3.74 (4.09) (4.93) at 32,000, 7.25 (7.30)
// (8.99) at 50,000, 13.5 (15.5) (14.9) at 70,000, 25.3 (25.8) (28.4) at 100,003,
// 193 (194) (198) at 300,000; 12 components 0.87 (1.10) at 16,384 and 2.94 (4.06)
// at 50,000.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "rerank.cuh"
#include "tc_ptx.cuh"
#include "topk.cuh"

namespace rsc {

namespace simtp {

constexpr int kQ = 128;                   // query rows per item, threads per CTA
static_assert(kQ == kTieItem && kQ <= 512, "ties items; 16 bits a hit");
constexpr int kR = 64;                    // database rows per tile
constexpr int kPitch = kR + 4;            // s rows on 16 bytes, conflict-free scans
// top-k buffer entries per thread: with 12 two CTAs share an SM at DP = 64 too
// (cap_of).  64 components, k = 15, one CTA with 20 entries and two with 12: rows
// without clusters 10.7 and 8.5 ms at 50,000 rows (full scan 8.7), 36.7 and 30.0 at
// 100,003 (31.7), 2.0 and 1.8 at 16,384 (1.6); clustered rows 2.09 and 1.74 at
// 100,003, 0.69 and 0.52 at 10,000, 0.88 and 0.92 at 16,384.
constexpr int kCapNarrow = 20, kCapWide = 12;
constexpr int kChunk = 256;               // tiles tested at a time
constexpr int kWords = kChunk / 32;
constexpr int kExactFirst = 2, kExactStep = 16;   // tiles between two looks at the bounds in the ties pass
constexpr int kSmallLeaf = 16;            // rows (see tile_table_kernel)
constexpr int kBatch = 1024;              // hits of the ties pass scored at a time
constexpr int kSeeds = 8;                 // nearest tiles scanned first when the window's do not bound an item
constexpr int kWin = 3;                   // tiles on each side of the query tile scanned first
constexpr int kStages = 2;
constexpr int kMaxCtas = 320;             // persistent CTAs at most
constexpr int kBigItems = 640;            // items that may be split
constexpr int kSegs = 16;                 // parts of a split item at most
constexpr int kSegTiles = 16;             // tiles per part at least
constexpr int kUnits = 1792;              // lists (of kQ rows) of split items and their parts
constexpr uint32_t kSleepNs = 2000;                // suspend of a wait per try
constexpr long long kDrainBudget = 2000000000LL;   // ~1 s of SM clocks, for copies in flight when a CTA leaves

// tiles at most: every leaf may end in a partial one; an even number
__host__ __device__ inline int64_t tiles_max(int64_t n) { return (ceil_div(n, (int64_t)kR) + kOrderMaxLeaves + 2) / 2 * 2; }
// record of a tile: DP x 64 components, then 64 |y|^2
__host__ __device__ inline int record_floats(int DP) { return (DP + 1) * kR; }

static_assert(kBatch * (sizeof(unsigned long long) + sizeof(uint16_t)) <= 2 * kCapWide * kQ * sizeof(float),
              "the ties pass keeps its batch where the buffers lie");
__host__ __device__ inline int cap_of(int DP) { return DP <= 56 ? kCapNarrow : kCapWide; }

struct Smem {
    int xs, ys, s, buf, list, cen, bars, total;   // byte offsets
};
__host__ __device__ inline Smem smem_layout(int DP) {
    Smem m;
    m.xs = 0;                                             // query tile: two records' components
    m.ys = m.xs + 2 * DP * kR * 4;
    m.s = m.ys + kStages * record_floats(DP) * 4;
    m.buf = m.s + kQ * kPitch * 4;
    m.list = m.buf + 2 * cap_of(DP) * kQ * 4;
    m.cen = m.list + kChunk * 4;
    m.bars = m.cen + 2 * 64 * 4;
    m.total = m.bars + 256;
    return m;
}

// ------------------------------------------------------------------ packing

// The tiles: tile_pos[t] = first sorted position, tile_rows[t] = rows; *T =
// their number.  Successive leaves form a run unless their centroids are
// further apart than twice the sum of their mean squared radii; runs are cut
// into tiles of 64.  Rows far from everything often have a leaf each, and so a
// tile each, which is scanned like a full one: where that would make the tiles a
// quarter more, two small leaves are not cut apart.  (50 components, clusters and
// 2.5 % strays far off: 50,000 rows 11.7 ms with all cuts, 6.8 so, 7.3 by the full
// scan; 200,000 rows 116, 74 and 95; 24,000 rows with 1 %: 3.3, 1.5 and 2.7.  With
// 0.2 % the cuts stay and pay, 50,000 rows 2.5 to 4.2 ms: a stray's own tile is
// soon dropped.)
// One block, two leaves (then two runs) per thread.
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
    bool small[2];   // a cut between two small leaves
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int l = 2 * tid + h;
        cut[h] = 0;
        small[h] = false;
        if (l < lv.count && pos[l + 1] > pos[l]) {
            int p = l - 1;
            while (p >= 0 && pos[p + 1] == pos[p]) --p;   // the last leaf with rows
            cut[h] = 1;
            if (p >= 0) {
                const float *a = lv.cent + (int64_t)cid[l] * DP, *b = lv.cent + (int64_t)cid[p] * DP;
                float d = 0.f;
                for (int t = 0; t < DP; ++t) d = fmaf(a[t] - b[t], a[t] - b[t], d);
                cut[h] = d > 2.f * (lv.var[cid[l]] + lv.var[cid[p]]) ? 1 : 0;
                small[h] = cut[h] && max(pos[l + 1] - pos[l], pos[p + 1] - pos[p]) < kSmallLeaf;
            }
        }
    }
    const int more = __syncthreads_count(small[0]) + __syncthreads_count(small[1]);
    if ((int64_t)more * 4 * kR > n) {   // uniform
        if (small[0]) cut[0] = 0;
        if (small[1]) cut[1] = 0;
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
            float *__restrict__ cenT, float *__restrict__ rad, float *__restrict__ nmax, int32_t *__restrict__ id_min) {
    __shared__ float ys[64][kR + 1];
    __shared__ float cen[64];
    __shared__ float red[2][8];
    __shared__ int first_id[8];
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
    const int own_id = r < rows ? (int32_t)o : INT_MAX, least = __reduce_min_sync(0xffffffffu, own_id);
    if (l == 0) ids[t * kR + r] = own_id;
    if ((tid & 31) == 0) first_id[tid >> 5] = least;
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
            first_id[0] = min(first_id[0], first_id[w]);
        }
        id_min[t] = first_id[0];
        rad[t] = rows > 0 ? sqrtf(md) * (1.f + 0x1p-10f) + 1e-6f : -1.f;   // -1: an empty tile
        nmax[t] = mn;
    }
}

// --------------------------------------------------------------------- top-k

// The KC smallest s of one query in registers (RowTopK), fed through a
// per-thread shared-memory buffer as BufferedTopK is, with the row's bound as
// the filter.  Equal values beyond the list's end are dropped whatever their
// ids: such a row is finished by the ties pass.  That is settled once a list is
// full of entries within reach of its k-th, and from then on it takes in only
// what lies below the k-th (rows that are all the same would otherwise buffer
// every value they meet).
template <int KC, int kCap>
struct List {
    RowTopK<KC> top;
    float bound;          // values above it cannot be among the k nearest, or are left to the ties pass:
    float floor;          // values from here on may have been left out
    float vv, v2;         // |y_i|^2 and |y_i|
    uint32_t sbase;
    int cnt, k, w;

    __device__ __forceinline__ void start(float nn, int k_, int w_) {
        top.init();
#pragma unroll
        for (int c = 0; c < KC; ++c) top.key[c] = FLT_MAX;   // finite: infinite values are never accepted
        bound = FLT_MAX;
        floor = INFINITY;
        vv = nn;
        v2 = sqrtf(nn);
        cnt = 0;
        k = k_;
        w = w_;
    }
    __device__ __forceinline__ float reach_of(float t) const { return rr::reach(t, vv, v2, w); }
    __device__ __forceinline__ float kth() const {
        float t = top.key[0];
#pragma unroll
        for (int c = 1; c < KC; ++c) t = fmaxf(t, c < k ? top.key[c] : -FLT_MAX);   // ascending: the k-th
        return t;
    }
    __device__ __forceinline__ float reach() const { return reach_of(kth()); }
    // The list is final: its last key tells what was left out.  A last entry
    // within the reach of the final k-th then means that the list is short of
    // some row.
    __device__ __forceinline__ void finish() {
        if (floor <= reach()) top.key[KC - 1] = fminf(top.key[KC - 1], floor);
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
    // Between two scans: whether the row is one for the ties pass by now.
    __device__ __forceinline__ void settle() {
        const float t = kth();
        if (top.id[KC - 1] >= 0 && top.thr() <= reach_of(t) && t < floor) {
            floor = t;
            bound = fminf(bound, below(t));
        }
    }
    static __device__ __forceinline__ float below(float t) {   // the next smaller float
        const int b = __float_as_int(t);
        return __int_as_float(t > 0.f ? b - 1 : t < 0.f ? b + 1 : (int)0x80000001);
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
    const int32_t *id_min;  // smallest row id of a tile
    int64_t n, stride;      // rows; stride of cenT (tiles_max)
    int DP, width, k;
    float beta;
    int32_t *cand;          // [n, KC] positions, -1 for none
    int32_t *tie_items;     // items with rows for the ties pass
    float *tie_bound;       // [item * kQ + row] their reach (-inf: not such a row), items on the list only
    int *tie_count, *counter;
    int *tie_done;          // parts of a tie item that are done
    uint32_t *bits;         // [CTAs][stride / 32] tiles an item keeps
    int32_t *big;           // [kBigItems][1 + kSeeds] items to be split, their seeds (-1 pads)
    int *big_count, *unit;  // their number (may exceed big_cap), next part
    float *big_bound;       // [kBigItems * kQ] their rows' bounds
    int *heavy, *light;     // items that kept many tiles (ties aside), and items done that kept few
    int slots;              // CTAs that are resident at once
    int64_t units;          // lists there is room for
    int big_cap;            // entries of `big` at most: two lists each at least
    int *tie_unit;          // next part of a tie item
    // split: [units][kQ][KC], the lists of parts (position in `big`, part) from the
    // front and the items' own, in that order, from the back
    float *part_key;        // flat: [query slots][part_segs][KC] lists of the parts; a slot is a query
    int32_t *part_id;       // tile pair's (split: position in `big`; flat: item) kQ rows
    int part_segs;
    float *vv;              // [query slots] |y|^2 (flat)
    unsigned long long *scanned;   // tiles scanned (a statistic)
    unsigned int *status;
    long long wait_budget;         // SM clocks a wait for a copy may take (tc_wait_budget)
};

// Parts of each of `count` items over `tiles` tiles: as many as cost least, waves
// of CTAs times a part's tiles (about three more for its start), while there is
// room for them (own: lists an item takes besides its parts').
__device__ __forceinline__ int part_count(const Args &g, int64_t count, int64_t tiles, int own) {
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int s = 1; s <= kSegs && (s == 1 || (count * (s + own) <= g.units && tiles >= (int64_t)s * kSegTiles)); ++s) {
        const int64_t c = ceil_div(count * s, (int64_t)g.slots) * (ceil_div(tiles, (int64_t)s) + 3);
        if (c < cost) {
            cost = c;
            best = s;
        }
    }
    return best;
}

// The candidates of an item's rows (a thread each; lists finished), and the
// item for the ties pass if more rows may lie within reach of one than its list
// holds (cut: a part's list was short).
template <int KC, int kCap>
__device__ __forceinline__ void emit(const Args &g, const List<KC, kCap> &tk, int64_t item, int tid, bool live, bool cut) {
    const float reach = tk.reach();
    if (live) {
        int32_t *out = g.cand + (g.tile_pos[2 * item + (tid >> 6)] + (tid & 63)) * (int64_t)KC;
#pragma unroll
        for (int c = 0; c < KC; ++c) {
            out[c] = tk.top.key[c] <= reach ? tk.top.id[c] : -1;   // -1 also where empty
        }
    }
    const bool tie = live && (cut || (tk.top.id[KC - 1] >= 0 && tk.top.key[KC - 1] <= reach));
    if (__syncthreads_or(tie)) {
        g.tie_bound[item * kQ + tid] = tie ? reach : -INFINITY;
        if (tid == 0) g.tie_items[atomicAdd(g.tie_count, 1)] = (int32_t)item;
    }
}

// ---------------------------------------------------------------------- ties

// The ties pass: the rows of the items on the tie list once more, against the
// tiles that their bounds keep, in the tiled search's own way; a value within
// a row's bound is a hit.  The block scores a tile's hits together, a thread each,
// with the re-rank's arithmetic (one row may have all of them), and a thread takes
// the scores of its own row into the k smallest (distance, id).  A row's list full of zeros
// needs no larger id any more, scored or not, and a tile whose smallest id
// is past those of all rows is left out: equal rows end after a few tiles.
// What it costs, whole calls, k = 15 (in brackets a warp per row over all
// tiles, hits scored one by one; then the full scan, which drops ties beyond its
// lists): 100,000 equal rows 2.9 ms (about 1,500; 25.8), 20,000 of them 2.2 (58;
// 1.4); 100,000 rows of one component 2.8 (41; 9.5); 100,000 clustered rows of 50,
// 5 % of them in groups of 30 copies, 2.2 (18; 25.9); 50,000 rows of 50 zeros and
// ones, which no sphere separates, 10.4 (31; 7.3).  The worst is a row as far from
// most others: 99,990 copies of a row and ten others 33 ms (25.9).
template <int KE>
struct Exact {
    static constexpr unsigned long long kNone = 0x7f8000007fffffffull;   // (+inf, INT_MAX)
    unsigned long long best[KE];   // (bits of the squared distance, id), ascending
    float bound;                   // -inf: nothing is wanted
    float vv, v2, beta;            // |y_i|^2 and |y_i|; what s leaves out of a squared distance besides
    int w;

    __device__ __forceinline__ void start(float bound_, float nn, float beta_, int w_) {
#pragma unroll
        for (int c = 0; c < KE; ++c) best[c] = kNone;
        bound = bound_;
        vv = nn;
        v2 = sqrtf(nn);
        beta = beta_;
        w = w_;
    }
    __device__ __forceinline__ void insert(unsigned long long v) {
        if (!(v < best[KE - 1])) return;
#pragma unroll
        for (int c = KE - 1; c > 0; --c) best[c] = v < best[c - 1] ? best[c - 1] : v < best[c] ? v : best[c];
        if (v < best[0]) best[0] = v;
        // a row at a squared distance D has s within e of D - vv - beta
        if (best[KE - 1] < kNone)
            bound = fminf(bound, rr::reach(__uint_as_float((unsigned)(best[KE - 1] >> 32)) - vv - beta, vv, v2, w));
    }
    // nothing but zeros with smaller ids than this one
    __device__ __forceinline__ bool full_before(int id) const { return best[KE - 1] <= (unsigned)id; }
};

// What the ties pass scores and where it puts it.
struct TieArgs {
    const float *R;   // the re-rank's rows, by position
    int64_t rs;
    int d;
    bool cosine, vec;
    int32_t *idx;
    float *dist;

    // (squared distance, id) of the rows at positions a and b, `id` the one of b
    __device__ __forceinline__ unsigned long long score(int64_t a, int64_t b, int id) const {
        const float *x = R + a * rs, *y = R + b * rs;
        float key = rr::dist2_thread(x, y, d, cosine, vec);
        if (cosine) {
            const bool fx = x[d] != 0.f, fy = y[d] != 0.f;   // rows of zeros
            if (fx || fy) key = (fx && fy) ? 0.f : 2.f;
        }
        return (unsigned long long)__float_as_uint(key) << 32 | (unsigned)id;
    }
};

// kWhole: an item per query tile pair.  An item that keeps more than 1 / 16 of
// the tiles (a tile that holds a row far from its cluster, or spans two) would
// outlast all others on its CTA (100k rows: 10 ms for one); such items are put on
// a list with their rows' lists and bounds so far, as long as there is room, and
// kSplitItems runs the rest of them in parts, segments of the database, whose
// lists merge_kernel joins.  Where nearly all items are such (rows that no sphere
// separates) they are run at once as long as they fill whole waves of CTAs, and
// the last, partial wave is what is split.
// kFlat: rows in their own order, part_segs parts per item and no tests: the
// search of fewer rows than an ordering pays for (see launch_knn_simt_flat).
// kTies, kFlatTies: the ties pass after either search (KC: Exact's entries).
enum { kWhole, kSplitItems, kFlat, kTies, kFlatTies };
template <int KC, int kMode, int kCap>
__global__ void __launch_bounds__(kQ, 2) simt_pruned_kernel(const Args g, const TieArgs ta) {
    constexpr bool kSplit = kMode == kSplitItems, kIsFlat = kMode == kFlat || kMode == kFlatTies;
    constexpr bool kExact = kMode == kTies || kMode == kFlatTies;
    const int64_t tie_items = kExact ? *g.tie_count : 0;
    if (kExact && tie_items == 0) return;
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
    typename std::conditional<kExact, Exact<KC>, List<KC, kCap>>::type tk;
    if constexpr (!kExact) tk.sbase = (uint32_t)__cvta_generic_to_shared(reinterpret_cast<float *>(sm + m.buf) + tid);
    // bounded; a budget shorter than a few sleeps is polled
    const uint32_t sleep_ns = g.wait_budget < 8 * (long long)kSleepNs ? 0 : kSleepNs;
    auto wait = [&](uint64_t *bar, uint32_t parity, long long budget) -> bool {
        if (sleep_ns == 0 ? tc::mbar_test_wait(bar, parity) : tc::mbar_try_wait(bar, parity)) return true;
        const long long t0 = clock64();
        while (!tc::mbar_arrived(bar, parity, sleep_ns))
            if (clock64() - t0 > budget) {
                record_status(g.status, RSC_ERR_TIMEOUT);
                return false;
            }
        return true;
    };
    const int64_t tiles = *g.T;   // an odd count is followed by an empty tile
    const int64_t big_items = kSplit ? min(*g.big_count, g.big_cap) : 0;
    if (kSplit && big_items == 0) return;
    const int64_t seg_len = ceil_div(tiles, (int64_t)(kMode == kFlat ? g.part_segs
                                                      : kExact       ? part_count(g, tie_items, tiles, 0)
                                                      : kSplit       ? part_count(g, big_items, tiles, 1)
                                                                     : 1));
    const int segs = kMode == kFlat ? g.part_segs : (int)ceil_div(tiles, seg_len);
    const int64_t pairs = ceil_div(tiles, (int64_t)2);
    const int64_t units = kExact            ? tie_items * segs
                          : kMode == kFlat ? pairs * segs
                          : kSplit         ? big_items * segs
                                           : pairs;
    const int64_t whole_waves = pairs / g.slots * g.slots;
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
            if constexpr (kExact) {
                // this row's hits, and their places among the block's
                unsigned hit[2] = {0u, 0u};
                if (!tk.full_before(kIsFlat ? j0 : g.id_min[tt])) {   // (a row that wants nothing has no hits)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll 8
                        for (int c = 0; c < 32; c += 4) {
                            const float4 v = *reinterpret_cast<const float4 *>(sr + 32 * h + c);
                            hit[h] |= (v.x <= tk.bound ? 1u : 0u) << c | (v.y <= tk.bound ? 2u : 0u) << c |
                                      (v.z <= tk.bound ? 4u : 0u) << c | (v.w <= tk.bound ? 8u : 0u) << c;
                        }
                }
                int at = __popc(hit[0]) + __popc(hit[1]);
                const int mine = at;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, at, o);
                    if (lane >= o) at += y;
                }
                if (lane == 31) seeds[warp] = at;
                __syncthreads();
                int total = 0;
                at -= mine;
#pragma unroll
                for (int w = 0; w < kQ / 32; ++w) {
                    if (w < warp) at += seeds[w];
                    total += seeds[w];
                }
                unsigned long long *keys = reinterpret_cast<unsigned long long *>(sm + m.buf);   // [kBatch]
                uint16_t *pair = reinterpret_cast<uint16_t *>(keys + kBatch);                    // row, column
                const int32_t *tile_ids = g.ids + (int64_t)tt * kR;
                int end = at;   // hits of this row listed so far
                for (int b0 = 0; b0 < total; b0 += kBatch) {
                    const int from = end;
                    for (; (hit[0] | hit[1]) != 0 && end < b0 + kBatch; ++end) {
                        const int h = hit[0] != 0 ? 0 : 1, c = __ffs(h ? hit[1] : hit[0]) - 1;
                        if (h) hit[1] &= hit[1] - 1;
                        else hit[0] &= hit[0] - 1;
                        pair[end - b0] = tk.full_before(tile_ids[32 * h + c]) ? 0xffffu : (uint16_t)(tid << 6 | 32 * h | c);
                    }
                    __syncthreads();
                    for (int x = tid; x < min(kBatch, total - b0); x += kQ) {
                        const int rc = pair[x], row = rc >> 6, c = rc & 63;
                        keys[x] = rc == 0xffff ? Exact<KC>::kNone
                                               : ta.score(seeds[4 + (row >> 6)] + (row & 63), j0 + c, tile_ids[c]);
                    }
                    __syncthreads();
                    for (int x = from; x < end; ++x) tk.insert(keys[x - b0]);
                    __syncthreads();   // the lists and seeds may be rewritten
                }
                if (total == 0) __syncthreads();
                continue;
            } else {
            if (first && i == 0 && g.tile_rows[tt] == kR) tk.start_bound(sr);   // a full tile, empty lists
#pragma unroll 1
            for (int h = 0; h < kR; h += 8) {
                const float4 lo = *reinterpret_cast<const float4 *>(sr + h), hi = *reinterpret_cast<const float4 *>(sr + h + 4);
                const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                tk.offer8(v, j0 + h);
            }
            }
        }
        scanned += nl;
        if constexpr (!kExact) {
            tk.flush();
            if constexpr (kMode != kFlat) tk.settle();   // (a flat part is one scan, or a few)
        }
        __syncthreads();   // the list may be rewritten
        return true;
    };
    for (;; ++items) {
        __syncthreads();
        if (tid == 0) *item_s = atomicAdd(kExact ? g.tie_unit : kSplit ? g.unit : g.counter, 1);
        __syncthreads();
        const int64_t unit = *item_s;
        if (unit >= units) break;
        const int32_t *big = g.big + unit / segs * (1 + kSeeds);   // kSplit
        const int64_t item = kExact ? (int64_t)g.tie_items[unit / segs] : kSplit ? (int64_t)big[0] : kIsFlat ? unit / segs : unit;
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
        bool live = (tid & 63) < g.tile_rows[2 * item + (tid >> 6)];
        float nn = 0.f;
        const float *xr = xs + (tid >> 6) * DP * kR + (tid & 63);
        for (int t = 0; t < g.width; ++t) nn = fmaf(xr[t * kR], xr[t * kR], nn);
        if constexpr (kExact) {
            tk.start(live ? g.tie_bound[item * kQ + tid] : -INFINITY, nn, g.beta, g.width);
            live = tk.bound > -INFINITY;
            if (tid < 2) seeds[4 + tid] = g.tile_pos[2 * item + tid];   // (read after the next barriers)
        } else {
            tk.start(nn, g.k, g.width);
        }
        float rq[2] = {0.f, 0.f}, nq[2] = {0.f, 0.f};
        if (!kIsFlat) {
            rq[0] = g.rad[2 * item];
            rq[1] = g.rad[2 * item + 1];
            nq[0] = g.nmax[2 * item];
            nq[1] = g.nmax[2 * item + 1];
        }
        const int wlo = kExact ? 0 : (int)max((int64_t)0, 2 * item - kWin);
        const int whi = kExact ? 0 : (int)min(tiles, 2 * item + 2 + kWin);
        // the range of tiles in chunks, from the chunk of the query tiles on
        const int64_t lo = kMode != kWhole ? min(tiles, (unit % segs) * seg_len) : 0;
        const int64_t hi = kMode != kWhole ? min(tiles, lo + seg_len) : tiles;
        const int chunks = (int)ceil_div(hi - lo, (int64_t)kChunk), c0 = kMode != kWhole ? 0 : (int)((2 * item) / kChunk);
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
        // A part of a split item and an item of the ties pass, whose bounds are
        // known, have kChunks only.
        enum { kWindow, kMark, kNearest, kAgain, kChunks };
        int step = kMode == kWhole ? kWindow : kChunks, ci = 0, n_seeds = 0;
        int64_t kept = 0;
        float near_d[2] = {INFINITY, INFINITY}, tq[2] = {INFINITY, INFINITY};
        int near_t[2] = {-1, -1};
        bool fresh = true, all_ties = false;   // fresh: tq must be taken anew
        int deferred = -1;                     // place on the list of items to be split
        if (kSplit) {
            if (tid < kSeeds) seeds[tid] = big[1 + tid];
            while (n_seeds < kSeeds && big[1 + n_seeds] >= 0) ++n_seeds;
            if constexpr (kSplit) tk.bound = live ? g.big_bound[unit / segs * kQ + tid] : -INFINITY;
        }
        int64_t done = 0;   // flat, exact: tiles of the part seen so far
        bool first = !kSplit;
        // exact: rows of ids from here on are wanted by no row (INT_MAX: some may be)
        auto last_id = [&]() -> int {
            unsigned v = 0;
            if constexpr (kExact) v = !live ? 0u : tk.best[KC - 1] <= 0xffffffffull ? (unsigned)tk.best[KC - 1] : (unsigned)INT_MAX;
            v = __reduce_max_sync(0xffffffffu, v);
            if (lane == 0) seeds[warp] = (int)v;
            __syncthreads();
            const int most_id = max(max(seeds[0], seeds[1]), max(seeds[2], seeds[3]));
            __syncthreads();
            return most_id;
        };
        int id_end = INT_MAX;
        while (true) {
            int nl = 0;
            if (kIsFlat) {   // the part's tiles, from the query's own on when they are among them
                const int64_t len = hi - lo, from = !kExact && 2 * item >= lo && 2 * item < hi ? 2 * item - lo : 0;
                nl = (int)min((int64_t)(!kExact ? kChunk : first ? kExactFirst : kExactStep), len - done);
                if (nl <= 0) break;
                if (kExact && (lo + done) * kR >= last_id()) break;   // uniform; ids ascend
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
                if (kExact ? lo + done >= hi : ci == chunks) {
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
                    if constexpr (kMode == kWhole) {
                        // many tiles, and most rows are for the ties pass already:
                        // all of them, with the bounds they have
                        if (kept > most && step == kAgain &&
                            16 * __syncthreads_count(live && tk.floor < INFINITY) >= __syncthreads_count(live)) {
                            all_ties = true;
                            break;
                        }
                    }
                    if (kept > most && step == kAgain) {
                        if (tid == 0) {
                            const int h = atomicAdd(g.heavy, 1), l = *reinterpret_cast<volatile int *>(g.light);
                            const bool now = unit < whole_waves && h >= 8 && h >= 4 * l;
                            const int at = now ? g.big_cap : atomicAdd(g.big_count, 1);
                            *item_s = at < g.big_cap ? at : -1;
                            if (*item_s >= 0) {
                                g.big[at * (1 + kSeeds)] = (int32_t)item;
                                for (int x = 0; x < kSeeds; ++x) g.big[at * (1 + kSeeds) + 1 + x] = seeds[x];
                            }
                        }
                        __syncthreads();
                        deferred = *item_s;
                        if (deferred >= 0) break;
                    }
                    step = kChunks;
                    continue;
                }
                const int chunk = c0 + ci < chunks ? c0 + ci : c0 + ci - chunks;
                const int64_t base = kExact ? lo + done : lo + (int64_t)chunk * kChunk;
                uint32_t *word = bits + chunk * kWords;
                ++ci;
                const bool all = kMode != kWhole || step == kMark;
                if (!all) {
                    uint32_t any = 0;
#pragma unroll
                    for (int x = 0; x < kWords; ++x) any |= word[x];
                    if (any == 0) continue;
                }
                if (fresh) {   // the tiles' bounds (dead rows ask for nothing)
                    float tau = live ? tk.bound + nn : -INFINITY;
                    if (live && !(tau < INFINITY)) tau = INFINITY;   // also NaN
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) tau = fmaxf(tau, __shfl_xor_sync(0xffffffffu, tau, o));
                    if (lane == 0) redf[warp] = tau;
                    __syncthreads();
                    tq[0] = fmaxf(redf[0], redf[1]);
                    tq[1] = fmaxf(redf[2], redf[3]);
                    if (kExact) id_end = last_id();
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
                        if (kExact) keep &= g.id_min[t] < id_end;
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
                    if (kExact) {   // few at a time, fewer at first: the bounds fall quickly
                        const int few = first ? kExactFirst : kExactStep;
                        __syncthreads();
                        done += nl > few ? list[few - 1] + 1 - base : (int64_t)kChunk;
                        nl = min(nl, few);
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
            if (step == kWindow) step = kMark;
            else if (step == kNearest) {
                step = kAgain;
                kept = 0;
            }
        }
        if constexpr (kExact) {
            // parts leave their lists to the one that is done last
            const int64_t pos = unit / segs;
            bool last = true;
            if (segs > 1) {
                unsigned long long *lists = reinterpret_cast<unsigned long long *>(g.part_key);
                auto list_of = [&](int64_t u) { return lists + (u * kQ + tid) * KC; };
                if (live)
#pragma unroll
                    for (int c = 0; c < KC; ++c) __stcg(list_of(unit) + c, tk.best[c]);
                __threadfence();
                __syncthreads();
                if (tid == 0) *item_s = atomicAdd(g.tie_done + pos, 1) == segs - 1;
                __syncthreads();
                last = *item_s != 0;
                if (last && live) {
                    __threadfence();
                    for (int64_t u = pos * segs; u < (pos + 1) * segs; ++u)
                        for (int c = 0; u != unit && c < KC; ++c) {
                            const unsigned long long v = __ldcg(list_of(u) + c);
                            if (!(v < tk.best[KC - 1])) break;   // ascending
                            tk.insert(v);
                        }
                }
            }
            if (last && live) {
                const int64_t o = (int64_t)g.ids[item * kQ + tid] * g.k;
#pragma unroll
                for (int c = 0; c < KC; ++c)
                    if (c < g.k) {
                        const int id = (int)(unsigned)tk.best[c];
                        const float d2 = __uint_as_float((unsigned)(tk.best[c] >> 32));
                        ta.idx[o + c] = id != INT_MAX ? id : -1;
                        ta.dist[o + c] = id != INT_MAX ? (ta.cosine ? 0.5f * d2 : sqrtf(d2)) : INFINITY;
                    }
            }
        } else {
            if constexpr (kMode != kFlat) tk.finish();
            if (kMode != kWhole || deferred >= 0) {   // uniform
                const int64_t at = kIsFlat  ? ((item * kQ + tid) * g.part_segs + unit % segs) * KC
                                   : kSplit ? (unit * kQ + tid) * KC
                                            : ((g.units - 1 - deferred) * kQ + tid) * KC;
                if (live) {
                    float *pk = g.part_key + at;
                    int32_t *pi = g.part_id + at;
#pragma unroll
                    for (int c = 0; c < KC; c += 4) {
                        *reinterpret_cast<float4 *>(pk + c) =
                            make_float4(tk.top.key[c], tk.top.key[c + 1], tk.top.key[c + 2], tk.top.key[c + 3]);
                        *reinterpret_cast<int4 *>(pi + c) =
                            make_int4(tk.top.id[c], tk.top.id[c + 1], tk.top.id[c + 2], tk.top.id[c + 3]);
                    }
                    if (kIsFlat && unit % segs == 0) g.vv[item * kQ + tid] = nn;
                    if (kMode == kWhole) g.big_bound[deferred * kQ + tid] = tk.bound;
                }
            } else {
                if (tid == 0 && kept <= most) atomicAdd(g.light, 1);
                emit(g, tk, item, tid, live, all_ties);
            }
        }
    }
    if (!kExact && tid == 0 && scanned) atomicAdd(g.scanned, scanned);
}

// Joins the lists of a split item and its parts.
template <int KC>
__global__ void __launch_bounds__(kQ) merge_kernel(const Args g) {
    const int64_t b = blockIdx.x, count = min(*g.big_count, g.big_cap);
    if (b >= count) return;
    const int64_t tiles = *g.T;
    const int64_t segs = ceil_div(tiles, ceil_div(tiles, (int64_t)part_count(g, count, tiles, 1)));
    const int tid = threadIdx.x;
    const int64_t item = g.big[b * (1 + kSeeds)];
    const bool live = (tid & 63) < g.tile_rows[2 * item + (tid >> 6)];
    const float *xr = g.rec + (2 * item + (tid >> 6)) * record_floats(g.DP) + (tid & 63);
    float nn = 0.f;
    for (int t = 0; t < g.width; ++t) nn = fmaf(xr[t * kR], xr[t * kR], nn);
    List<KC, kCapWide> tk;   // (no buffer is used)
    tk.start(nn, g.k, g.width);
    auto list_at = [&](int64_t s) { return ((s < segs ? b * segs + s : g.units - 1 - b) * kQ + tid) * KC; };   // segs: the item's own
    for (int64_t s = segs; live && s >= 0; --s) {
        const int64_t at = list_at(s);
#pragma unroll 1
        for (int c = 0; c < KC; ++c) {
            const float v = g.part_key[at + c];
            const int j = g.part_id[at + c];
            if (j < 0 || !(v < tk.top.thr())) break;   // ascending
            tk.top.insert(v, j);
        }
    }
    // a part's full list whose last key is within reach is short of some rows
    const float reach = tk.reach();
    bool cut = false;
    for (int64_t s = 0; live && s <= segs; ++s) {
        const int64_t at = list_at(s) + KC - 1;
        cut |= g.part_id[at] >= 0 && g.part_key[at] <= reach;
    }
    emit(g, tk, item, tid, live, cut);
}

constexpr int kCounters = 10;
constexpr int kMaxList = 40;

// Parts' lists: the keys, then the ids (or Exact's entries in the whole of it).
template <class L>
void take_lists(Carve &cv, L &l, size_t entries) {
    l.part_key = reinterpret_cast<float *>(cv.take<unsigned long long>(entries));
    l.part_id = reinterpret_cast<int32_t *>(l.part_key + entries);
}

struct Layout {
    float *rec, *cenT, *rad, *nmax, *tie_bound;
    int32_t *ids, *tile_pos, *tile_rows, *tie_items, *id_min;
    int *counters;   // tie_count, counter, scanned (64 bits), tiles, big_count, unit, tie_unit, heavy, light; tie_done follows
    int64_t zeroed;  // ints
    int32_t *big, *part_id;
    uint32_t *bits;
    float *part_key, *big_bound;
    int64_t units;
    size_t bytes;
};
Layout layout(void *scratch, int64_t n, int DP, int k) {
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
    L.id_min = cv.take<int32_t>((size_t)tiles);
    L.tie_items = cv.take<int32_t>((size_t)tiles / 2);
    L.tie_bound = cv.take<float>((size_t)tiles * kR);
    L.zeroed = kCounters + tiles / 2;
    L.counters = cv.take<int>((size_t)L.zeroed);
    L.big = cv.take<int32_t>(kBigItems * (1 + kSeeds));
    L.big_bound = cv.take<float>(kBigItems * kQ);
    L.bits = cv.take<uint32_t>((size_t)kMaxCtas * ceil_div(tiles, (int64_t)kChunk) * kWords);
    // room for eight parts of every item of a small input, of up to 1,792 lists in
    // all: 30 MB at 16,384 rows, 44 MB from 25,000 on (k <= 16; 50 and 73 beyond)
    L.units = std::min<int64_t>(kUnits, 9 * (ceil_div(n, (int64_t)kQ) + 8));
    take_lists(cv, L, (size_t)L.units * simt_pruned_list(k) * kQ);
    L.bytes = cv.used;
    return L;
}

constexpr int kCtasPerSm = 2;   // resident

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
    g.id_min = L.id_min;
    g.tie_items = L.tie_items;
    g.tie_bound = L.tie_bound;
    g.tie_count = L.counters;
    g.tie_unit = L.counters + 7;
    g.tie_done = L.counters + kCounters;
    g.counter = L.counters + 1;
    g.scanned = reinterpret_cast<unsigned long long *>(L.counters + 2);
    g.bits = L.bits;
    g.big = L.big;
    g.big_count = L.counters + 5;
    g.unit = L.counters + 6;
    g.part_key = L.part_key;
    g.part_id = L.part_id;
    g.part_segs = 0;
    g.heavy = L.counters + 8;
    g.light = L.counters + 9;
    g.big_bound = L.big_bound;
    g.units = L.units;
    g.big_cap = (int)std::min<int64_t>(kBigItems, L.units / 2);
    g.slots = kCtasPerSm * sm_count();
    g.vv = nullptr;
    g.status = status;
    g.wait_budget = tc_wait_budget();
    return g;
}

}  // namespace simtp

// Entries beyond k: enough that rows within rounding of the k-th hardly ever
// fill the list.
int simt_pruned_list(int k) { return k <= 16 ? 24 : k <= 32 ? 40 : 0; }

size_t simt_pruned_scratch_bytes(int64_t n, int DP, int k) { return simtp::layout(nullptr, n, DP, k).bytes; }

const unsigned long long *simt_pruned_scanned(void *scratch, int64_t n, int DP, int k) {
    return reinterpret_cast<unsigned long long *>(simtp::layout(scratch, n, DP, k).counters + 2);
}

namespace simtp {

template <int KC>
cudaError_t launch_list(const Args &g, int64_t tiles, cudaStream_t st) {
    const int smem = smem_layout(g.DP).total;
    const bool wide = cap_of(g.DP) == kCapWide;
    auto whole = wide ? simt_pruned_kernel<KC, kWhole, kCapWide> : simt_pruned_kernel<KC, kWhole, kCapNarrow>;
    auto split = wide ? simt_pruned_kernel<KC, kSplitItems, kCapWide> : simt_pruned_kernel<KC, kSplitItems, kCapNarrow>;
    cudaError_t e = cudaFuncSetAttribute(whole, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(split, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    whole<<<(unsigned)std::min<int64_t>(tiles / 2, std::min(kMaxCtas, kCtasPerSm * sm_count())), kQ, smem, st>>>(g, TieArgs{});
    split<<<(unsigned)(kCtasPerSm * sm_count()), kQ, smem, st>>>(g, TieArgs{});
    merge_kernel<KC><<<kBigItems, kQ, 0, st>>>(g);
    return cudaGetLastError();
}

template <int kMode>
cudaError_t launch_ties(const Args &g, int d, int metric, const float *R, int64_t rs, int32_t *idx, float *dist,
                        cudaStream_t st) {
    const bool vec = rs % 4 == 0 && reinterpret_cast<uintptr_t>(R) % 16 == 0;
    const TieArgs ta{R, rs, d, metric == RSC_COSINE, vec, idx, dist};
    const int smem = smem_layout(g.DP).total;
    auto kern = g.k <= 16 ? simt_pruned_kernel<16, kMode, kCapWide> : simt_pruned_kernel<32, kMode, kCapWide>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)(kCtasPerSm * sm_count()), kQ, smem, st>>>(g, ta);
    return cudaGetLastError();
}

}  // namespace simtp

OrderTarget simt_pruned_target() { return {128, true}; }

cudaError_t launch_knn_simt_pruned(const float *Y, const float *ny, int64_t n, int DP, int width, int k, int metric,
                                   const int32_t *perm, const OrderLeaves &leaves, void *scratch, int32_t *cand,
                                   unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    const Layout L = layout(scratch, n, DP, k);
    const int64_t tiles = tiles_max(n);
    cudaError_t e = cudaMemsetAsync(L.counters, 0, L.zeroed * sizeof(int), st);
    if (e != cudaSuccess) return e;
    tile_table_kernel<<<1, 1024, 0, st>>>(leaves, n, DP, L.tile_pos, L.tile_rows, L.counters + 4);
    pack_kernel<<<(unsigned)tiles, 256, 0, st>>>(Y, ny, DP, perm, tiles, L.tile_pos, L.tile_rows, L.counters + 4, L.rec,
                                                 L.ids, L.cenT, L.rad, L.nmax, L.id_min);
    const Args g = make_args(L, n, DP, width, k, metric, cand, status);
    return simt_pruned_list(k) == 24 ? launch_list<24>(g, tiles, st) : launch_list<kMaxList>(g, tiles, st);
}

cudaError_t launch_simt_ties(int64_t n, int d, int DP, int width, int k, int metric, void *scratch, const float *R,
                             int64_t rs, int32_t *idx, float *dist, unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    const Args g = make_args(layout(scratch, n, DP, k), n, DP, width, k, metric, nullptr, status);
    return launch_ties<kTies>(g, d, metric, R, rs, idx, dist, st);
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

constexpr int kFlatCounters = 6;

struct FlatLayout {
    float *rec, *part_key, *vv, *tie_bound;
    int32_t *ids, *tile_pos, *tile_rows, *part_id, *tie_items;
    int *counters;   // tie_count, counter, scanned (64 bits), tiles, tie_unit; tie_done and tie_flag follow
    int64_t zeroed;  // ints
    size_t bytes;
};
FlatLayout flat_layout(void *scratch, int64_t n, int DP, int k) {
    Carve cv(scratch);
    FlatLayout L;
    const int64_t items = ceil_div(n, (int64_t)kQ);
    const size_t parts = (size_t)items * kQ * simt_flat_segs(n) * simt_pruned_list(k);
    L.rec = cv.take<float>((size_t)items * 2 * record_floats(DP));
    L.ids = cv.take<int32_t>((size_t)items * kQ);
    L.tile_pos = cv.take<int32_t>((size_t)items * 2);
    L.tile_rows = cv.take<int32_t>((size_t)items * 2);
    take_lists(cv, L, parts);
    L.vv = cv.take<float>((size_t)items * kQ);
    L.tie_items = cv.take<int32_t>((size_t)items);
    L.tie_bound = cv.take<float>((size_t)items * kQ);
    L.zeroed = kFlatCounters + 2 * items;
    L.counters = cv.take<int>((size_t)L.zeroed);
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
    g.part_segs = simt_flat_segs(n);
    g.vv = L.vv;
    g.tie_items = L.tie_items;
    g.tie_bound = L.tie_bound;
    g.tie_unit = L.counters + 5;
    g.tie_done = L.counters + kFlatCounters;
    // lists of 16 (k <= 16) or 32 entries in the room of part_segs lists an item
    g.units = ceil_div(n, (int64_t)kQ) * g.part_segs;
    g.slots = kCtasPerSm * sm_count();
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
int simt_flat_segs(int64_t n) {
    const int64_t items = ceil_div(n, (int64_t)simtp::kQ), tiles = ceil_div(n, (int64_t)simtp::kR);
    const int64_t slots = kPlanSMs * simtp::kCtasPerSm;
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
    return {L.part_key, L.part_id, L.vv, simt_flat_segs(n), simt_pruned_list(k), L.counters,
            L.counters + simtp::kFlatCounters + ceil_div(n, (int64_t)simtp::kQ), L.tie_items, L.tie_bound};
}

cudaError_t launch_knn_simt_flat(const float *Y, const float *ny, int64_t n, int DP, int width, int k, void *scratch,
                                 unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    const FlatLayout L = flat_layout(scratch, n, DP, k);
    const Args g = flat_args(L, n, DP, width, k, status);
    cudaError_t e = cudaMemsetAsync(L.counters, 0, L.zeroed * sizeof(int), st);
    if (e != cudaSuccess) return e;
    const int64_t items = ceil_div(n, (int64_t)kQ);
    pack_flat_kernel<<<(unsigned)(2 * items), 256, 0, st>>>(Y, ny, n, DP, L.rec, L.ids, L.tile_pos, L.tile_rows,
                                                           L.counters + 4);
    const int smem = smem_layout(DP).total;
    const bool wide = cap_of(DP) == kCapWide;
    auto kern = simt_pruned_list(k) == 24
                    ? (wide ? simt_pruned_kernel<24, kFlat, kCapWide> : simt_pruned_kernel<24, kFlat, kCapNarrow>)
                    : (wide ? simt_pruned_kernel<kMaxList, kFlat, kCapWide> : simt_pruned_kernel<kMaxList, kFlat, kCapNarrow>);
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
    kern<<<(unsigned)std::min<int64_t>(items * g.part_segs, kCtasPerSm * sm_count()), kQ, smem, st>>>(g, TieArgs{});
    return cudaGetLastError();
}

cudaError_t launch_simt_flat_ties(int64_t n, int d, int DP, int width, int k, int metric, void *scratch, const float *R,
                                  int64_t rs, int32_t *idx, float *dist, unsigned int *status, cudaStream_t st) {
    using namespace simtp;
    Args g = flat_args(flat_layout(scratch, n, DP, k), n, DP, width, k, status);
    g.beta = metric == RSC_COSINE ? 1.f : 0.f;
    return launch_ties<kFlatTies>(g, d, metric, R, rs, idx, dist, st);
}

}  // namespace rsc
