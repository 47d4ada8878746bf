// pond_mlp_train.cuh -- training kernels of the learned face-gauge predictor (forward, loss
// and backward through the activations and the weight gradients; Adam), on the tcgen05 tensor cores.
#pragma once

#include "pond_mlp.cuh"

namespace pond {
namespace mlp {

// Forward pass of 128 rows: x [n][ldx] features, out [n][16].
__global__ void __launch_bounds__(kThreads)
forward_kernel(const float *prm, const float *x, int ldx, long long n, float *out, unsigned int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    const long long row = (long long)blockIdx.x * kRows + threadIdx.x;
    const bool valid = row < n;
    if (threadIdx.x < 32) tc::tmem_alloc(&tmem_base, 128);
    if (threadIdx.x == 0) tc::mbar_init(&mbar, 1);
    stage_weights(prm, sm);
    for (int k = 0; k < kIn; ++k) put_bf16(sm + sA1, threadIdx.x, k, kIn, valid ? x[row * ldx + k] : 0.f);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base;
    uint32_t phase = 0;
    float o[kOutP];
    const bool ok = forward_tile(prm, sm, tmem, &mbar, phase, o);
    if (valid && ok)
        for (int j = 0; j < kOutP; ++j) out[row * kOutP + j] = o[j];
    if (!ok && threadIdx.x == 0) atomicOr(err, 1u);
    drain(&mbar, phase, ok);
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) tc::tmem_free(tmem, 128);
}

// Loss and gradient of a batch.  A CTA takes `per` tiles of 128 rows and keeps everything between x
// and its share of the gradient on the SM: the activations and their gradients stay in shared
// memory as BF16, and each tile's weight gradients
//   dW1 += dZ1^T X, dW2 += dZ2^T H1, dW3 += dOut^T H2
// accumulate in tensor memory over the CTA's tiles.  A matrix that one GEMM reads K-major (row = sample)
// the weight gradients read MN-major (K = sample) from the same bytes: a core matrix of 8 samples
// x 8 units is the same 128 bytes both ways, only the descriptor's strides differ.  X carries a
// column of ones and dZ1, dZ2 lie side by side as one 128-unit operand, so that column of dW1
// gives both bias gradients; dOut has three columns in use and is summed by the threads.
// Each CTA writes its partial gradient; grad_reduce_kernel adds them in a fixed order.
//
// Two threads a row (each half of the columns), two CTAs per SM (113 KB of shared memory and 256
// columns of tensor memory each), so that one's GEMM waits cover the other's element-wise work.
//
// Measured (GB300, 65536 rows): 21 us and 3.9 for the sum, against 192 us for a kernel that wrote the
// activations with two-byte stores and 355 us for one that read them back and transposed them element by
// element.  Bound by latency: staging the weights, then six dependent GEMMs with the work between
// them for each of two tiles a CTA (reading x alone takes 2 us).
constexpr int kGradThreads = 256;
constexpr int kGradMaxCtas = 304;
constexpr int kPartStride = kParams + 4;        // a partial gradient, then the partial loss
constexpr int kXw = 64, kZw = 128;              // columns of X with its ones, of [dZ1 | dZ2]
constexpr int gX = 0;                           // X | 1    [128][64]
constexpr int gH1 = gX + kRows * kXw * 2;       // H1       [128][64]
constexpr int gH2 = gH1 + kRows * kHid * 2;     // H2       [128][64]
constexpr int gZ = gH2 + kRows * kHid * 2;      // dZ1|dZ2  [128][128]
constexpr int gO = gZ + kRows * kZw * 2;        // dOut     [128][16]
constexpr int gW1 = gO + kRows * kOutP * 2;     // W1       [64][48]
constexpr int gW2 = gW1 + kHid * kIn * 2;       // W2       [64][64]
constexpr int gW3 = gW2 + kHid * kHid * 2;      // W3       [16][64]
constexpr int gW3t = gW3 + kOutP * kHid * 2;    // W3^T     [64][16]
constexpr int gW2t = gW3t + kHid * kOutP * 2;   // W2^T     [64][64]
constexpr int kGradSmem = gW2t + kHid * kHid * 2;
// an MN-major operand of fewer than 128 units is read past its units: that stays inside the plan
static_assert(gO + (15 * 2 + 15) * 128 + 128 <= kGradSmem && gZ + 15 * 2048 + 8 * 128 + 15 * 128 + 128 <= kGradSmem,
              "the weight gradients' operands lie within the shared memory");

// B operand from a row-major matrix W [rows][K] (or, t, its transpose: row k of W is column k)
__device__ __forceinline__ void stage_matrix(const float *W, unsigned char *dst, int rows, int K, bool t)
{
    for (int e = threadIdx.x; e < rows * (K / 8); e += kGradThreads) {
        const int r = t ? e % rows : e / (K / 8), k0 = 8 * (t ? e / rows : e % (K / 8));
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = t ? W[(k0 + i) * rows + r] : W[r * K + k0 + i];
        put_bf16x8(dst, r, k0, K, v);
    }
}

__global__ void __launch_bounds__(kGradThreads, 2)
grad_kernel(const float *prm, const float *x, int ldx, const float *y, int ldy, long long n, int per, float *part,
            unsigned int *err)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ float bias[2 * kHid + kOutP], sums[4][kOut + 1];
    const int tid = threadIdx.x, half = tid >> 7, r = tid & 127;
    if (tid < 32) tc::tmem_alloc(&tmem_base, 256);
    if (tid == 0) tc::mbar_init(&mbar, 1);
    stage_matrix(prm + oW1, sm + gW1, kHid, kIn, false);
    stage_matrix(prm + oW2, sm + gW2, kHid, kHid, false);
    stage_matrix(prm + oW3, sm + gW3, kOutP, kHid, false);
    stage_matrix(prm + oW3, sm + gW3t, kHid, kOutP, true);
    stage_matrix(prm + oW2, sm + gW2t, kHid, kHid, true);
    for (int e = tid; e < 2 * kHid + kOutP; e += kGradThreads)
        bias[e] = prm[e < kHid ? ob1 + e : e < 2 * kHid ? ob2 + e - kHid : ob3 + e - 2 * kHid];
    if (half == 0) {   // X's columns 48 .. 63: one, zeros
        const float one[8] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, none[8] = {};
        put_bf16x8(sm + gX, r, kIn, kXw, one);
        put_bf16x8(sm + gX, r, kIn + 8, kXw, none);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_base, lane = uint32_t(r & ~31) << 16;
    const uint32_t tW1 = tmem + 64, tW2 = tmem + 128, tW3 = tmem + 192;   // columns 0 .. 63: the tile's GEMMs
    uint32_t phase = 0;
    // GEMMs over what has been stored, waited for by every thread; false on time-out
    auto run = [&](auto &&issue) {
        tc::fence_smem_to_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {
            issue();
            tc::commit(&mbar);
        }
        const bool ok = __syncthreads_and(tc::mbar_wait(&mbar, phase, kPolls)) != 0;
        if (ok) phase ^= 1u;
        tc::fence_after_sync();
        return ok;
    };
    const int c0 = half * 32;   // this thread's columns
    auto read32 = [&](float *v) {
        tc::tmem_ld16(tmem + lane + c0, v);
        tc::tmem_ld16(tmem + lane + c0 + 16, v + 16);
    };
    const bool vec = ldx % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    const float inv = float(kOut * n);
    float lsum = 0.f, bsum[kOut] = {};
    const long long tiles = (n + kRows - 1) / kRows;
    const long long t_begin = (long long)blockIdx.x * per, t_end = min(t_begin + per, tiles);
    bool ok = true;
    for (long long t = t_begin; t < t_end && ok; ++t) {
        const long long row0 = t * kRows, row = row0 + r;
        const bool valid = row < n, first = t == t_begin;
        float target[kOut] = {};
        if (half == 0 && valid)
#pragma unroll
            for (int j = 0; j < kOut; ++j) target[j] = y[row * ldy + kIn + j];
        // eight neighbouring threads store the eight rows of a core matrix
        for (int e = tid; e < kRows * (kIn / 8); e += kGradThreads) {
            const int q = e >> 3, rr = (q / (kIn / 8)) * 8 + (e & 7), k0 = 8 * (q % (kIn / 8));
            float v[8] = {};
            if (row0 + rr < n) {
                const float *src = x + (row0 + rr) * ldx + k0;
                if (vec) {
                    const float4 a = reinterpret_cast<const float4 *>(src)[0], b = reinterpret_cast<const float4 *>(src)[1];
                    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
                    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) v[i] = src[i];
                }
            }
            put_bf16x8(sm + gX, rr, k0, kXw, v);
        }
        float v[32];
        // hidden layers (rows past the batch store zeros: they add nothing to the weight gradients)
#pragma unroll 1
        for (int layer = 0; layer < 2 && ok; ++layer) {
            ok = run([&] {
                if (layer == 0) tc::gemm_issue(tmem, sm + gX, kXw, sm + gW1, kIn, kIn, kHid);
                else tc::gemm_issue(tmem, sm + gH1, kHid, sm + gW2, kHid, kHid, kHid);
            });
            if (!ok) break;
            read32(v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = valid ? fmaxf(v[j] + bias[layer * kHid + c0 + j], 0.f) : 0.f;
#pragma unroll
            for (int k = 0; k < 32; k += 8) put_bf16x8(sm + (layer ? gH2 : gH1), r, c0 + k, kHid, v + k);
        }
        if (!ok) break;
        ok = run([&] { tc::gemm_issue(tmem, sm + gH2, kHid, sm + gW3, kHid, kHid, kOutP); });
        if (!ok) break;
        if (half == 0) {
            // dL/dout for L = sum (out - y)^2 / (3 n)
            float d[kOutP] = {};
            tc::tmem_ld16(tmem + lane, v);
#pragma unroll
            for (int j = 0; j < kOut; ++j) {
                const float e = valid ? v[j] + bias[2 * kHid + j] - target[j] : 0.f;
                d[j] = 2.f * e / inv;
                lsum += e * e;
                bsum[j] += __bfloat162float(__float2bfloat16_rn(d[j]));
            }
            put_bf16x8(sm + gO, r, 0, kOutP, d);
            put_bf16x8(sm + gO, r, 8, kOutP, d + 8);
        }
        // dH2 = dOut W3, dZ2 = dH2 * [h2 > 0]; then the same one layer down
#pragma unroll 1
        for (int layer = 1; layer >= 0 && ok; --layer) {
            ok = run([&] {
                if (layer == 1) {
                    tc::gemm_issue(tmem, sm + gO, kOutP, sm + gW3t, kOutP, kOutP, kHid);
                    tc::gemm_issue_mn(tW3, sm + gO, kOutP, sm + gH2, kHid, kRows, kHid, !first);
                } else {
                    tc::gemm_issue(tmem, sm + gZ + 8 * 128, kZw, sm + gW2t, kHid, kHid, kHid);
                    tc::gemm_issue_mn(tW2, sm + gZ + 8 * 128, kZw, sm + gH1, kHid, kRows, kHid, !first);
                }
            });
            if (!ok) break;
            read32(v);
#pragma unroll
            for (int k = 0; k < 32; k += 8) {
                float h[8];
                get_bf16x8(sm + (layer ? gH2 : gH1), r, c0 + k, kHid, h);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[k + i] = h[i] > 0.f ? v[k + i] : 0.f;
                put_bf16x8(sm + gZ, r, (layer ? kHid : 0) + c0 + k, kZw, v + k);
            }
        }
        if (!ok) break;
        ok = run([&] { tc::gemm_issue_mn(tW1, sm + gZ, kZw, sm + gX, kXw, kRows, kXw, !first); });
    }
    if (ok) {
        // units 0 .. 63 of dW1 with b1 in column 48, b2 in the same column of units 64 .. 127
        float *o = part + size_t(blockIdx.x) * kPartStride;
        auto put_row = [&](float *dst, uint32_t col, int chunks) {
            float w[16];
            for (int c = 0; c < chunks; ++c) {
                tc::tmem_ld16(col + lane + 16 * c, w);
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4 *>(dst + 16 * c + i) = make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]);
            }
        };
        if (half == 0) {
            float w[16];
            if (r < kHid) put_row(o + oW1 + r * kIn, tW1, kIn / 16);
            tc::tmem_ld16(tW1 + lane + kIn, w);
            o[r < kHid ? ob1 + r : ob2 + r - kHid] = w[0];
            float q[kOut + 1] = {bsum[0], bsum[1], bsum[2], lsum / inv};
#pragma unroll
            for (int j = 0; j <= kOut; ++j) {
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) q[j] += __shfl_down_sync(0xffffffffu, q[j], s);
                if ((tid & 31) == 0) sums[tid >> 5][j] = q[j];
            }
        } else if (r < kHid) {
            put_row(o + oW2 + r * kHid, tW2, kHid / 16);
            // (whole warps take the tensor-memory loads)
            float w[16];
            if (r < 32)
                for (int c = 0; c < kHid / 16; ++c) {
                    tc::tmem_ld16(tW3 + lane + 16 * c, w);
                    if (r < kOutP)
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            *reinterpret_cast<float4 *>(o + oW3 + r * kHid + 16 * c + i) = make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]);
                }
        }
        __syncthreads();
        if (tid <= kOutP) {   // the bias of the outputs (three in use), then the loss
            const int j = tid < kOut ? tid : kOut;
            const float s = sums[0][j] + sums[1][j] + sums[2][j] + sums[3][j];
            o[ob3 + tid] = tid < kOut || tid == kOutP ? s : 0.f;
        }
    } else if (tid == 0) {
        atomicOr(err, 1u);
    }
    drain(&mbar, phase, ok);
    tc::fence_before_sync();
    __syncthreads();
    if (tid < 32) tc::tmem_free(tmem, 256);
}

// grad[p] = sum of part[c][p] over the CTAs c, 32 parameters a block: eight warps take every eighth
// CTA, then add up in order, so the result does not depend on scheduling.  The last column
// adds to the loss.  Nothing on an error (the call reports POND_ERR_TIMEOUT).
__global__ void __launch_bounds__(256) grad_reduce_kernel(const float *part, int nparts, float *grad, float *loss, const unsigned int *err)
{
    __shared__ float acc[8][32];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, p = blockIdx.x * 32 + l;
    if (*(const volatile unsigned int *)err) return;
    float a = 0.f;
    if (p <= kParams) {
#pragma unroll 8
        for (int c = w; c < nparts; c += 8) a += part[size_t(c) * kPartStride + p];
    }
    acc[w][l] = a;
    __syncthreads();
    if (w == 0 && p <= kParams) {
#pragma unroll
        for (int i = 1; i < 8; ++i) a += acc[i][l];
        if (p < kParams) grad[p] = a;
        else *loss += a;
    }
}

__global__ void adam_kernel(float *prm, const float *g, float *m, float *v, float lr, float b1, float b2, float eps,
                            float bc1, float bc2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    const float gi = g[i];
    m[i] = b1 * m[i] + (1.f - b1) * gi;
    v[i] = b2 * v[i] + (1.f - b2) * gi * gi;
    prm[i] -= lr * (m[i] / bc1) / (sqrtf(v[i] / bc2) + eps);
}

}  // namespace mlp
}  // namespace pond
