// Warp-wide ascending sort of (key, id) pairs held in registers.
//
// E pairs per lane; element v = e * 32 + lane of a virtual array of 32 * E.
// A bitonic network: strides >= 32 compare a lane's own elements, smaller
// strides exchange with lane ^ stride through shuffles.  Order: key, then id
// (the exact-kNN tie rule).  Every lane of the warp must call it.
#pragma once

#include "common.cuh"

namespace rsc {

__device__ __forceinline__ bool pair_gt(float ka, int ia, float kb, int ib) {
    return ka > kb || (ka == kb && ia > ib);
}

template <int E>
__device__ __forceinline__ void warp_sort_pairs(float (&key)[E], int (&id)[E]) {
    const int lane = threadIdx.x & 31;
    constexpr int P = 32 * E;
#pragma unroll
    for (int size = 2; size <= P; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
                const int es = stride >> 5;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int pe = e ^ es;
                    if (pe > e) {
                        const bool asc = (((e << 5) | lane) & size) == 0;
                        if (pair_gt(key[e], id[e], key[pe], id[pe]) == asc) {
                            const float tk = key[e];
                            key[e] = key[pe];
                            key[pe] = tk;
                            const int ti = id[e];
                            id[e] = id[pe];
                            id[pe] = ti;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const float pk = __shfl_xor_sync(0xffffffffu, key[e], stride);
                    const int pi = __shfl_xor_sync(0xffffffffu, id[e], stride);
                    const bool asc = (((e << 5) | lane) & size) == 0;
                    const bool lower = (lane & stride) == 0;
                    // the lower position of an ascending pair keeps the smaller pair
                    const bool take =
                        (lower == asc) ? pair_gt(key[e], id[e], pk, pi) : pair_gt(pk, pi, key[e], id[e]);
                    if (take) {
                        key[e] = pk;
                        id[e] = pi;
                    }
                }
            }
        }
    }
}

// The 32 smallest of two ascending runs, one pair per lane each, into (bk, bi):
// elementwise minima of one and the other reversed form a bitonic run, sorted
// by five half-cleaners.
__device__ __forceinline__ void warp_merge_best(float &bk, int &bi, float key, int id) {
    const int lane = threadIdx.x & 31;
    const float rk = __shfl_xor_sync(0xffffffffu, key, 31);
    const int ri = __shfl_xor_sync(0xffffffffu, id, 31);
    if (pair_gt(bk, bi, rk, ri)) {
        bk = rk;
        bi = ri;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float pk = __shfl_xor_sync(0xffffffffu, bk, o);
        const int pi = __shfl_xor_sync(0xffffffffu, bi, o);
        const bool lower = (lane & o) == 0;
        if (lower ? pair_gt(bk, bi, pk, pi) : pair_gt(pk, pi, bk, bi)) {
            bk = pk;
            bi = pi;
        }
    }
}

}  // namespace rsc
