// Tensor-core GEMM for the partitioner network (BF16 operands, FP32
// accumulation in tensor memory), sm_103a.
//
//   C[m, n] = sum_k A(m, k) B(k, n) (+ bias[n]),
//   A(m, k) = A[m * sam + k * sak],  B(k, n) = B[k * sbk + n * sbn]
//
// Operands come in FP32 with arbitrary strides (the forward pass multiplies
// activations by weights, the backward pass transposed gradients by
// activations), are passed through ReLU where asked and rounded to BF16 while
// the CTA's 128 threads stage them into shared memory in the K-major
// 128-byte-swizzled layout the tensor core reads (one 16-byte chunk of 8 k
// per store; consecutive threads take consecutive rows, so a stride-1 row or
// column dimension is read coalesced either way).  One thread issues
// tcgen05.mma M = 128, N = TN, K = 16 into a TN-column TMEM accumulator; two
// shared-memory stages let the next K block be staged while the tensor core
// consumes the current one.  Every warp reads its 32 TMEM lanes back with
// tcgen05.ld, adds the bias and stores its rows of C.  Every wait is bounded.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace rsc {
namespace mlp {

constexpr int kTM = 128;                              // C rows per CTA (TMEM lanes)
constexpr int kThreads = 128;
constexpr long long kWaitBudget = 2000000000LL;       // ~1 s of SM clocks
enum { kReluA = 4, kReluB = 8 };                       // same bits as the partitioner's GEMM flags

__device__ __forceinline__ uint8_t *align1024(uint8_t *p) {
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Byte offset of 16-byte chunk `ch` (k = 8 ch .. 8 ch + 7) of row r in a
// K-major tile of 128-byte rows under the 128-byte swizzle (8-row groups
// 1024 bytes apart, chunk index XOR row-in-group).
__device__ __forceinline__ uint32_t swz128(int r, int ch) {
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((ch ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, unsigned int *status) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!tc::mbar_try_wait_sleep(bar, parity, 2000)) {
        if (clock64() - t0 > kWaitBudget) {
            record_status(status, RSC_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// Rows [r0, r0 + R) x k block kc of an operand X(row, k) = X[row * s_row + k * s_k]
// staged as BF16 into a swizzled tile.
template <int R>
__device__ __forceinline__ void stage_tile(uint8_t *tile, const float *__restrict__ X, int64_t s_row, int64_t s_k,
                                           int r0, int rows, int k0, int K, bool relu) {
#pragma unroll 2
    for (int c = threadIdx.x; c < R * 8; c += kThreads) {
        const int r = c % R, ch = c / R;
        const int row = r0 + r, k = k0 + 8 * ch;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float x = 0.f;
            if (row < rows && k + e < K) x = X[(int64_t)row * s_row + (int64_t)(k + e) * s_k];
            v[e] = relu ? fmaxf(x, 0.f) : x;
        }
        *reinterpret_cast<uint4 *>(tile + swz128(r, ch)) =
            make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    }
}

template <int TN>
__global__ void __launch_bounds__(kThreads)
tc_gemm_kernel(int M, int N, int K, const float *__restrict__ A, int64_t sam, int64_t sak,
               const float *__restrict__ B, int64_t sbk, int64_t sbn, float *__restrict__ C, int64_t ldc,
               const float *__restrict__ bias, int flags, unsigned int *status) {
    constexpr int kABytes = kTM * 128, kBBytes = TN * 128, kStage = kABytes + kBBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = align1024(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + 2 * kStage);   // [2] stage read, [1] all MMAs done
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * kTM, n0 = blockIdx.x * TN;
    if (tid == 0) {
        tc::mbar_init(&bars[0], 1);
        tc::mbar_init(&bars[1], 1);
        tc::mbar_init(&bars[2], 1);
        tc::fence_barrier_init();
    }
    if (warp == 0) tc::tmem_alloc<TN>(tmem_slot);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    constexpr uint32_t idesc = tc::idesc_bf16_f32(kTM, TN);
    const int nk = (K + 63) / 64;
    for (int kc = 0; kc < nk; ++kc) {
        const int b = kc & 1;
        uint8_t *sa = smem + b * kStage;
        // the MMAs that last read this stage (K block kc - 2) must be done
        bool ok = kc < 2 || wait_bar(&bars[b], ((kc - 2) >> 1) & 1, status);
        if (!__syncthreads_and(ok)) break;
        stage_tile<kTM>(sa, A, sam, sak, m0, M, kc * 64, K, (flags & kReluA) != 0);
        stage_tile<TN>(sa + kABytes, B, sbn, sbk, n0, N, kc * 64, K, (flags & kReluB) != 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // staged bytes visible to the tensor core
        __syncthreads();
        if (tid == 0) {
            tc::tc_fence_after();
            const uint32_t a_addr = tc::smem_u32(sa), b_addr = tc::smem_u32(sa + kABytes);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                tc::mma_bf16(tmem, tc::smem_desc_sw128(a_addr + kk * 32), tc::smem_desc_sw128(b_addr + kk * 32),
                             idesc, (kc | kk) != 0);
            tc::mma_commit(&bars[b]);
        }
    }
    // every MMA issued so far has completed once bars[2] completes its phase
    if (tid == 0) tc::mma_commit(&bars[2]);
    const bool done = wait_bar(&bars[2], 0, status);
    tc::tc_fence_after();
    if (__syncthreads_and(done)) {
        const int r = warp * 32 + lane, m = m0 + r;
        const uint32_t lane_bits = (uint32_t)(warp * 32) << 16;
#pragma unroll 1
        for (int c0 = 0; c0 < TN; c0 += 32) {
            float v[32];
            __syncwarp();
            tc::tmem_ld32(tmem + lane_bits + c0, v);
            tc::tmem_wait_ld();
            if (m < M) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const int nn = n0 + c0 + j;
                    if (nn < N) C[(int64_t)m * ldc + nn] = v[j] + (bias ? bias[nn] : 0.f);
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc<TN>(tmem);
}

template <int TN>
cudaError_t launch(cudaStream_t st, int M, int N, int K, const float *A, int64_t sam, int64_t sak, const float *B,
                   int64_t sbk, int64_t sbn, float *C, int64_t ldc, const float *bias, int flags,
                   unsigned int *status) {
    constexpr int kSmem = 2 * (kTM * 128 + TN * 128) + 64 + 1024;
    auto kern = tc_gemm_kernel<TN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)ceil_div(N, TN), (unsigned)ceil_div(M, kTM));
    kern<<<grid, kThreads, kSmem, st>>>(M, N, K, A, sam, sak, B, sbk, sbn, C, ldc, bias, flags, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- routing
//
// The whole network d -> H -> H -> P and the R largest logits of every row in
// one persistent kernel, for H <= 256.  The GEMMs of one 128-row tile are far
// too small to fill the chip one at a time and their activations would pass
// through memory in FP32 (48 GEMM and 16 selection launches, 9.46 ms for 500k
// rows, H = 256, P = 512; this kernel 0.69 ms, bound by the epilogue's scan
// for the largest logits).  Here a CTA keeps a tile's
// activations in shared memory: the layers' accumulators alternate between
// two 256-column halves of TMEM, the epilogue adds the bias, applies ReLU,
// rounds to BF16 and writes the next layer's A operand in the layout the
// tensor core reads, and the logits never leave the SM.  Weights come as
// 32 KB blocks (256 outputs x 64 inputs, BF16, already swizzled by
// pack_weights_kernel) through a ring of bulk copies that runs ahead of the
// layers; they stay in L2 across tiles.  The multiply-accumulates of an
// output run in the same order (64-wide K blocks of four K = 16 steps) on the
// same rounded operands as in tc_gemm_kernel, so the logits are the same bits.
//   warps 0-7   epilogue: warp w reads TMEM lane quarter w & 3, columns
//               128 (w >> 2) .. + 127 of a half; a thread owns half a row
//   warp 8      weight blocks (one thread)
//   warp 9      MMA issue (one thread)
//   warps 10-11 the next tile's rows of X as the first layer's A operand
namespace route {

constexpr int kN = 256;                  // outputs per weight block (accumulator columns)
constexpr int kBlock = kN * 128;         // bytes of one weight block
constexpr int kABlock = kTM * 128;       // bytes of one 64-wide K block of an A operand
constexpr int kStages = 4;
constexpr int kEpi = 256;                // epilogue threads
constexpr int kStagers = 64;
constexpr int kThreads = kEpi + 64 + kStagers;
constexpr int kMaxP = 1024;
constexpr int kBias = 2 * kN + kMaxP;    // floats of the padded biases
constexpr int kMaxR = 8;
constexpr uint32_t kSleepNs = 20000;     // suspend of a wait per try
constexpr int kOffX = 0;
constexpr int kOffH = kOffX + kABlock;
constexpr int kOffW = kOffH + 4 * kABlock;
constexpr int kOffBias = kOffW + kStages * kBlock;
constexpr int kOffMerge = kOffBias + kBias * 4;
constexpr int kOffBar = kOffMerge + kTM * kMaxR * 8;
constexpr int kSmem = kOffBar + 256 + 1024;
static_assert(kSmem <= 227 * 1024, "one CTA per SM");

__host__ __device__ inline int k_blocks(int H) { return (H + 63) / 64; }
__host__ __device__ inline int chunks(int P) { return (P + kN - 1) / kN; }
__host__ __device__ inline int weight_blocks(int H, int P) { return 1 + k_blocks(H) * (1 + chunks(P)); }

// Block b of the packed weights: b = 0: W1; then W2's K blocks; then for every
// 256 outputs of W3 its K blocks.  One thread per 16-byte piece; zeros past
// the matrices' ends.  The last grid row copies the biases, zero padded.
__global__ void __launch_bounds__(256)
pack_weights_kernel(int d, int H, int P, const float *__restrict__ W1, const float *__restrict__ b1,
                    const float *__restrict__ W2, const float *__restrict__ b2, const float *__restrict__ W3,
                    const float *__restrict__ b3, uint8_t *__restrict__ out, float *__restrict__ bias) {
    const int nb = weight_blocks(H, P), kb = k_blocks(H);
    const int b = blockIdx.y, e = blockIdx.x * 256 + threadIdx.x;   // kN * 8 pieces
    if (b == nb) {
        if (e < kBias) {
            float v = 0.f;
            if (e < kN) v = e < H ? b1[e] : 0.f;
            else if (e < 2 * kN) v = e - kN < H ? b2[e - kN] : 0.f;
            else v = e - 2 * kN < P ? b3[e - 2 * kN] : 0.f;
            bias[e] = v;
        }
        return;
    }
    const int n = e >> 3, ch = e & 7;
    const float *src;
    int row = n, rows, K, k;
    if (b == 0) {
        src = W1; rows = H; K = d; k = 8 * ch;
    } else if (b <= kb) {
        src = W2; rows = H; K = H; k = (b - 1) * 64 + 8 * ch;
    } else {
        const int x = b - 1 - kb;
        src = W3; rows = P; K = H; k = (x % kb) * 64 + 8 * ch;
        row = (x / kb) * kN + n;
    }
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = (row < rows && k + i < K) ? src[(int64_t)row * K + k + i] : 0.f;
    *reinterpret_cast<uint4 *>(out + (size_t)b * kBlock + swz128(n, ch)) =
        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}

// Barriers of the two accumulator halves count uses: use u of a half has
// parity u & 1.
template <int R>
__global__ void __launch_bounds__(kThreads, 1)
route_kernel(const float *__restrict__ X, const int32_t *__restrict__ rows, int64_t count, int d, int H, int P,
             const uint8_t *__restrict__ packed, const float *__restrict__ bias_g, int32_t *__restrict__ out,
             unsigned int *status, long long wait_budget) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = align1024(smem_raw);
    uint8_t *sX = smem + kOffX, *sH = smem + kOffH, *sW = smem + kOffW;
    float *bias = reinterpret_cast<float *>(smem + kOffBias);
    float *mkey = reinterpret_cast<float *>(smem + kOffMerge);
    int *mid = reinterpret_cast<int *>(mkey + kTM * kMaxR);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kOffBar);
    uint64_t *empty = full + kStages;
    uint64_t *acc_full = empty + kStages;   // [2]
    uint64_t *acc_empty = acc_full + 2;     // [2]
    uint64_t *x_full = acc_empty + 2;       // the tile's X operand is staged
    uint64_t *x_empty = x_full + 1;         // the first layer has read it
    uint64_t *h_full = x_empty + 1;         // a hidden layer's operand is written
    uint64_t *merge_full = h_full + 1;      // the upper halves' best logits are written
    uint64_t *merge_empty = merge_full + 1; // and read
    uint64_t *done = merge_empty + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&acc_full[b], 1);
            tc::mbar_init(&acc_empty[b], kEpi / 32);
        }
        tc::mbar_init(x_full, kStagers / 32);
        tc::mbar_init(x_empty, 1);
        tc::mbar_init(h_full, kEpi / 32);
        tc::mbar_init(merge_full, kEpi / 64);
        tc::mbar_init(merge_empty, kEpi / 64);
        tc::mbar_init(done, 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    for (int e = tid; e < kBias; e += kThreads) bias[e] = bias_g[e];
    if (warp == 9) tc::tmem_alloc<512>(tmem_slot);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int kb = k_blocks(H), nc = chunks(P), nb = weight_blocks(H, P);
    const int64_t tiles = ceil_div(count, (int64_t)kTM);

    // bounded; a budget shorter than a few sleeps is polled
    const uint32_t sleep_ns = wait_budget < 8 * (long long)kSleepNs ? 0 : kSleepNs;
    auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
        if (sleep_ns == 0 ? tc::mbar_test_wait(bar, parity) : tc::mbar_try_wait(bar, parity)) return true;
        const long long t0 = clock64();
        while (!tc::mbar_arrived(bar, parity, sleep_ns)) {
            if (*abort_flag) return false;
            if (clock64() - t0 > wait_budget) {
                *abort_flag = 1;
                record_status(status, RSC_ERR_TIMEOUT);
                return false;
            }
        }
        return true;
    };
    auto drain = [&](uint64_t *bar, uint32_t parity) {   // the default budget, whatever is set
        const long long t0 = clock64();
        while (!tc::mbar_try_wait(bar, parity))
            if (clock64() - t0 > kWaitBudget) {
                record_status(status, RSC_ERR_TIMEOUT);
                return;
            }
    };

    if (warp < 8) {
        // ------------------------------------------------------- epilogue
        const int half = warp >> 2, r = (warp & 3) * 32 + lane;
        const uint32_t t0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + half * 128;
        uint32_t use[2] = {0, 0}, no = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++no) {
            for (int layer = 0; layer < 2; ++layer) {   // half 0: first hidden layer, half 1: second
                ok = __all_sync(0xffffffffu, wait(&acc_full[layer], use[layer] & 1));
                if (!ok) break;
                ++use[layer];
                tc::tc_fence_after();
                const float *bs = bias + layer * kN + half * 128;
#pragma unroll 1
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    float v[32];
                    __syncwarp();
                    tc::tmem_ld32(t0 + layer * kN + c0, v);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        float a[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) a[i] = fmaxf(v[8 * g + i] + bs[c0 + 8 * g + i], 0.f);
                        const int col = half * 128 + c0 + 8 * g;
                        *reinterpret_cast<uint4 *>(sH + (col >> 6) * kABlock + swz128(r, (col & 63) >> 3)) =
                            make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]),
                                       pack_bf16(a[6], a[7]));
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // bytes visible to the tensor core
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    tc::mbar_arrive(&acc_empty[layer]);
                    tc::mbar_arrive(h_full);
                }
            }
            if (!ok) break;
            // logits: this thread's columns of every chunk in ascending order,
            // the R largest kept sorted (an equal later one stays behind).
            // Empty places hold NaN: !(z <= NaN), so that every number, -inf
            // too, goes before them with the one comparison per logit (686 us
            // for 500k rows; 660 us with empty places of -inf, which take no
            // logit of -inf)
            float bk[R];
            int bi[R];
#pragma unroll
            for (int x = 0; x < R; ++x) {
                bk[x] = NAN;
                bi[x] = 0x7fffffff;
            }
            for (int c = 0; c < nc; ++c) {
                const int b = c & 1;
                ok = __all_sync(0xffffffffu, wait(&acc_full[b], use[b] & 1));
                if (!ok) break;
                ++use[b];
                tc::tc_fence_after();
                const int col0 = c * kN + half * 128;
#pragma unroll 1
                for (int c0 = 0; c0 < 128; c0 += 32) {
                    if (col0 + c0 >= P) break;   // warp-uniform
                    float v[32];
                    __syncwarp();
                    tc::tmem_ld32(t0 + b * kN + c0, v);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int col = col0 + c0 + j;
                        const float z = v[j] + bias[2 * kN + col];
                        if (col < P && !(z <= bk[R - 1])) {
                            if (z != z) continue;
#pragma unroll
                            for (int x = R - 1; x > 0; --x) {
                                const bool up = !(z <= bk[x - 1]), here = !(z <= bk[x]);
                                bi[x] = up ? bi[x - 1] : (here ? col : bi[x]);
                                bk[x] = up ? bk[x - 1] : (here ? z : bk[x]);
                            }
                            if (!(z <= bk[0])) {
                                bk[0] = z;
                                bi[0] = col;
                            }
                        }
                    }
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&acc_empty[b]);
            }
            if (!ok) break;
            // the two halves of a row: value descending, id ascending
            if (half == 1) {
                if (!(ok = __all_sync(0xffffffffu, wait(merge_empty, (no & 1) ^ 1)))) break;
#pragma unroll
                for (int x = 0; x < R; ++x) {
                    mkey[r * R + x] = bk[x];
                    mid[r * R + x] = bi[x];
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(merge_full);
                continue;
            }
            if (!(ok = __all_sync(0xffffffffu, wait(merge_full, no & 1)))) break;
            const int64_t row = tile * kTM + r;
            int x = 0;   // head of the other half
#pragma unroll
            for (int o = 0; o < R; ++o) {
                const float zo = mkey[r * R + x];
                const int io = mid[r * R + x];
                const bool other = io != 0x7fffffff && (!(zo <= bk[0]) || (zo == bk[0] && io < bi[0]));
                if (row < count) out[row * R + o] = other ? io : bi[0];
                if (other) {
                    ++x;
                } else {
#pragma unroll
                    for (int y = 0; y < R - 1; ++y) {
                        bk[y] = bk[y + 1];
                        bi[y] = bi[y + 1];
                    }
                    bk[R - 1] = NAN;
                    bi[R - 1] = 0x7fffffff;
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(merge_empty);
        }
    } else if (warp == 8) {
        if (lane == 0) {
            // ------------------------------------------------ weight blocks
            uint32_t g = 0;   // blocks issued
            bool ok = true;
            for (int64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x)
                for (int b = 0; b < nb; ++b, ++g) {
                    const int s = g % kStages;
                    if (!(ok = wait(&empty[s], ((g / kStages) & 1) ^ 1))) break;
                    tc::mbar_arrive_expect_tx(&full[s], kBlock);
                    tc::bulk_load(sW + s * kBlock, packed + (size_t)b * kBlock, kBlock, &full[s]);
                }
            // every copy this thread started lands before the CTA exits, whichever role gave up
            for (uint32_t t = g > kStages ? g - kStages : 0; t < g; ++t) drain(&full[t % kStages], (t / kStages) & 1);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            // ------------------------------------------------------ MMA issue
            constexpr uint32_t idesc = tc::idesc_bf16_f32(kTM, kN);
            uint32_t g = 0, use[2] = {0, 0}, hid = 0, no = 0;
            bool ok = true;
            // accumulator half b <- K blocks 0 .. n - 1 of A at `a` times the next n weight blocks
            auto layer = [&](int b, const uint8_t *a, int n) -> bool {
                if (!wait(&acc_empty[b], (use[b] & 1) ^ 1)) return false;
                ++use[b];
                for (int k = 0; k < n; ++k, ++g) {
                    const int s = g % kStages;
                    if (!wait(&full[s], (g / kStages) & 1)) return false;
                    tc::tc_fence_after();
                    const uint32_t a_addr = tc::smem_u32(a + k * kABlock), b_addr = tc::smem_u32(sW + s * kBlock);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc::mma_bf16(tmem + b * kN, tc::smem_desc_sw128(a_addr + kk * 32),
                                     tc::smem_desc_sw128(b_addr + kk * 32), idesc, (k | kk) != 0);
                    tc::mma_commit(&empty[s]);
                }
                tc::mma_commit(&acc_full[b]);
                return true;
            };
            for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++no) {
                if (!(ok = wait(x_full, no & 1))) break;
                if (!(ok = layer(0, sX, 1))) break;
                tc::mma_commit(x_empty);
                if (!(ok = wait(h_full, hid++ & 1))) break;
                if (!(ok = layer(1, sH, kb))) break;
                if (!(ok = wait(h_full, hid++ & 1))) break;
                for (int c = 0; c < nc && ok; ++c) ok = layer(c & 1, sH, kb);
                if (!ok) break;
            }
            tc::mma_commit(done);
            drain(done, 0);
        }
    } else {
        // ------------------------------------------------- rows of X, BF16
        const int t = tid - (kEpi + 64);
        uint32_t no = 0;
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++no) {
            if (!__all_sync(0xffffffffu, wait(x_empty, (no & 1) ^ 1))) break;
#pragma unroll 2
            for (int c = t; c < kTM * 8; c += kStagers) {
                const int r = c >> 3, ch = c & 7;
                const int64_t i = tile * kTM + r;
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = 0.f;
                if (i < count) {
                    const float *x = X + (rows ? (int64_t)rows[i] : i) * d;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (8 * ch + e < d) v[e] = x[8 * ch + e];
                }
                *reinterpret_cast<uint4 *>(sX + swz128(r, ch)) =
                    make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                               pack_bf16(v[6], v[7]));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(x_full);
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 9) {
        __syncwarp();
        tc::tmem_dealloc<512>(tmem);
    }
}

}  // namespace route

}  // namespace mlp

bool mlp_route_supported(int d, int H, int P) { return d <= 64 && H <= mlp::route::kN && P <= mlp::route::kMaxP; }

size_t mlp_route_weight_bytes(int H, int P) {
    return (size_t)mlp::route::weight_blocks(H, P) * mlp::route::kBlock + sizeof(float) * mlp::route::kBias;
}

cudaError_t launch_mlp_route_pack(cudaStream_t st, int d, int H, int P, const float *W1, const float *b1,
                                  const float *W2, const float *b2, const float *W3, const float *b3, void *packed) {
    using namespace mlp::route;
    const int nb = weight_blocks(H, P);
    uint8_t *out = static_cast<uint8_t *>(packed);
    float *bias = reinterpret_cast<float *>(out + (size_t)nb * kBlock);
    pack_weights_kernel<<<dim3(kN * 8 / 256, (unsigned)nb + 1), 256, 0, st>>>(d, H, P, W1, b1, W2, b2, W3, b3, out, bias);
    return cudaGetLastError();
}

cudaError_t launch_mlp_route(cudaStream_t st, const float *X, const int32_t *rows, int64_t count, int d, int H, int P,
                             int R, const void *packed, int32_t *out, unsigned int *status) {
    using namespace mlp::route;
    if (count <= 0) return cudaSuccess;
    auto kern = R == 1 ? route_kernel<1> : R == 2 ? route_kernel<2> : R == 4 ? route_kernel<4> : route_kernel<8>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    const uint8_t *w = static_cast<const uint8_t *>(packed);
    const float *bias = reinterpret_cast<const float *>(w + (size_t)weight_blocks(H, P) * kBlock);
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(count, (int64_t)mlp::kTM), sm_count());
    kern<<<grid, kThreads, kSmem, st>>>(X, rows, count, d, H, P, w, bias, out, status, tc_wait_budget());
    return cudaGetLastError();
}

cudaError_t launch_tc_gemm(cudaStream_t st, int M, int N, int K, const float *A, int64_t sam, int64_t sak,
                           const float *B, int64_t sbk, int64_t sbn, float *C, int64_t ldc, const float *bias,
                           int flags, unsigned int *status) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (N > 128) return mlp::launch<256>(st, M, N, K, A, sam, sak, B, sbk, sbn, C, ldc, bias, flags, status);
    return mlp::launch<128>(st, M, N, K, A, sam, sak, B, sbk, sbn, C, ldc, bias, flags, status);
}

}  // namespace rsc
