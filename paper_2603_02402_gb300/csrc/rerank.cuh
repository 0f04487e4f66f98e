// The exact re-rank's arithmetic for one pair of rows: eight lanes, lane s
// holding components 4 s .. 4 s + 3 and 32 + 4 s .. 32 + 4 s + 3.
#pragma once

#include "common.cuh"

namespace rsc {
namespace rr {

// This lane's components of a row of d <= 64 floats: two 16-byte loads when
// rows start on 16-byte boundaries (vec), else scalar loads; the same values
// either way.  Loads stop at the last 4-aligned piece holding a component
// below d; the rest of that piece is zero padding except the cosine rows' flag
// at column d, which is cleared.
__device__ __forceinline__ void load8(const float *row, int s, int d, bool cosine, bool vec, float (&v)[8]) {
    if (vec) {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
        const float4 a = (4 * s < d) ? __ldg(r4 + s) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 b = (32 + 4 * s < d) ? __ldg(r4 + 8 + s) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = (4 * s + i < d) ? __ldg(row + 4 * s + i) : 0.f;
            v[4 + i] = (32 + 4 * s + i < d) ? __ldg(row + 32 + 4 * s + i) : 0.f;
        }
    }
    if (cosine) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if ((i < 4 ? 4 * s + i : 28 + 4 * s + i) == d) v[i] = 0.f;
    }
}

// A bound for the FP32 search: whatever has s = |y_j|^2 - 2 y_i.y_j above
// reach(t) is further by the re-rank than k rows at or below t, when k rows lie
// at or below t.  vv, v: |y_i|^2 and |y_i|, w: components (knn_simt_prune.cu
// derives it).
__device__ __forceinline__ float reach(float t, float vv, float v, int w) {
    const float far = v + sqrtf(fmaxf(t + vv, 0.f));   // |y_i| + distance
    const float e = 1.25f * 0x1p-24f * (float)(w + 20) * (2.f * v * far + far * far);
    return t + 2.f * e + 0x1p-22f * fabsf(t);
}

// The same distance by one thread alone: the eight partial sums one after the
// other, added in the order in which the lanes' shuffles add them.
__device__ __forceinline__ float dist2_thread(const float *x, const float *y, int d, bool cosine, bool vec) {
    float part[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        part[s] = 0.f;
        if (4 * s >= d) continue;   // uniform
        float a[8], b[8];
        load8(x, s, d, cosine, vec, a);
        load8(y, s, d, cosine, vec, b);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float diff = a[i] - b[i];
            part[s] = fmaf(diff, diff, part[s]);
        }
    }
    return ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
}

// Sum of squared differences of the two rows (every lane of the eight gets it).
__device__ __forceinline__ float dist2(const float (&x)[8], const float (&y)[8]) {
    float part = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float diff = x[i] - y[i];
        part = fmaf(diff, diff, part);
    }
    part += __shfl_xor_sync(0xffffffffu, part, 1);
    part += __shfl_xor_sync(0xffffffffu, part, 2);
    part += __shfl_xor_sync(0xffffffffu, part, 4);
    return part;
}

}  // namespace rr
}  // namespace rsc
