// cnn.cu -- kernels of the candidate classifier (arXiv 2606.27262,
// Sec. 3.2.2: a CNN scores each sifted candidate from two images, its
// dedispersed dynamic spectrum and its DM transform; two networks, one per
// image, fused multiplicatively into one probability).
//
// The convolutions of layers 1 to 4 and their gradients are in cnn_tc.cu; here:
//   conv0_kernel, conv0_wgrad_kernel   the one-channel first layer, directly
//   pool_head_kernel, head_back_kernel pooling and linear head, and back
//   fuse_loss_kernel    fused probability, loss and its derivative
//   bias_part_kernel, column_sums_kernel   bias gradients
//   adam_kernel         the update
//   features_raw_kernel DM-time images of subband dynamic spectra
//   normalise_kernel    frequency-time and DM-time images normalised to zero
//                       mean and unit variance, as bf16
//   extract_kernel      subband spectra of candidates from the staged beam
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "sp_cnn_internal.h"

namespace sp {
namespace {

__device__ __forceinline__ uint32_t s_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid) {
    const int n = valid ? 16 : 0;  // zero-fill outside the matrix
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s_addr(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Two fp32 lanes of a 64-bit register (one instruction, each lane rounded as by the scalar one).
__device__ __forceinline__ void add2(unsigned long long &a, unsigned long long b) {
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a) : "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// Layer 0 (one input channel, 3x3, stride 2, zero padding 1) of both branches
// (blockIdx.y) as a direct convolution: a thread computes the sixteen outputs
// of four neighbouring pixels in fp32 from the bf16 weights (every product
// exact), then adds the bias, applies the ReLU and rounds once to bf16.  Its
// floor is the write of the output (134 MB a branch at batch 256: 20 us).  Four
// pixels share each read of the weights, two outputs go to one fma.f32x2, and a
// warp's output leaves in contiguous stores: 68 us a branch with one pixel and
// 32 scattered bytes per thread, 51 us now.
constexpr int kConv0Out = 16;
__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__global__ void __launch_bounds__(256) conv0_kernel(const ConvPair p, int H, int lwo4, uint32_t quads, int Kp) {
    __shared__ __align__(16) float ws[9][kConv0Out];
    __shared__ float bs[kConv0Out];
    __shared__ __align__(16) uint4 out_s[256][8];
    const bool br = blockIdx.y;
    const __nv_bfloat16 *w = br ? p.w[1] : p.w[0];
    if (threadIdx.x < kConv0Out * 9) {
        const int co = threadIdx.x / 9, k = threadIdx.x - co * 9;
        ws[k][co] = __bfloat162float(w[co * Kp + k]);
    }
    if (threadIdx.x < kConv0Out) bs[threadIdx.x] = (br ? p.bias[1] : p.bias[0])[threadIdx.x];
    __syncthreads();
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;  // pixels 4g .. 4g + 3
    const uint32_t gc = min(g, quads - 1);                     // threads past the end repeat the last
    const int Ho = H / 2;
    const int wq = (int)(gc & ((1u << lwo4) - 1)), ho = (int)((gc >> lwo4) % (uint32_t)Ho);
    const size_t n = (gc >> lwo4) / (uint32_t)Ho;
    const __nv_bfloat16 *img = (br ? p.x[1] : p.x[0]) + n * H * H;
    unsigned long long acc[4][kConv0Out / 2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int j = 0; j < kConv0Out / 2; ++j) acc[q][j] = 0ull;
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
        const int h = 2 * ho - 1 + ky;  // < H: only the row above the image is missing
        float v[9];
        if (h >= 0) {  // columns 8 wq - 1 .. 8 wq + 7
            const __nv_bfloat16 *row = img + (size_t)h * H + 8 * wq;
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(row));
            const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
            v[0] = wq > 0 ? __bfloat162float(row[-1]) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {  // bf16 = the upper half of an fp32
                v[2 * i + 1] = __uint_as_float(xs[i] << 16);
                v[2 * i + 2] = __uint_as_float(xs[i] & 0xFFFF0000u);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = 0.f;
        }
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) {
            const ulonglong2 *w4 = reinterpret_cast<const ulonglong2 *>(ws[3 * ky + kx]);
            unsigned long long vv[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) vv[q] = pack2(v[2 * q + kx], v[2 * q + kx]);
#pragma unroll
            for (int j = 0; j < kConv0Out / 4; ++j) {
                const ulonglong2 wj = w4[j];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    fma2(acc[q][2 * j], vv[q], wj.x);
                    fma2(acc[q][2 * j + 1], vv[q], wj.y);
                }
            }
        }
    }
    // A warp's 4 KB of output goes through shared memory (16-byte pieces
    // swizzled by lane), so that its stores are contiguous.
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t o[kConv0Out / 2];
#pragma unroll
        for (int j = 0; j < kConv0Out / 2; ++j) {
            const float2 a = unpack2(acc[q][j]);
            const __nv_bfloat162 h =
                __floats2bfloat162_rn(fmaxf(a.x + bs[2 * j], 0.f), fmaxf(a.y + bs[2 * j + 1], 0.f));
            o[j] = *reinterpret_cast<const uint32_t *>(&h);
        }
        out_s[threadIdx.x][(2 * q) ^ (lane & 7)] = make_uint4(o[0], o[1], o[2], o[3]);
        out_s[threadIdx.x][(2 * q + 1) ^ (lane & 7)] = make_uint4(o[4], o[5], o[6], o[7]);
    }
    __syncwarp();
    const uint32_t g0 = g - lane;
    uint4 *dst = reinterpret_cast<uint4 *>((br ? p.y[1] : p.y[0]) + (size_t)g0 * 4 * kConv0Out);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int id = 32 * i + lane, from = id >> 3;
        if (g0 + from < quads) dst[id] = out_s[threadIdx.x - lane + from][(id & 7) ^ (from & 7)];
    }
}

// Layer 0's weight and bias gradients: part[branch][block][k * 16 + co] = sum of
// dz[p][co] * x[p at tap k] over the block's pixels (k = 9: of dz alone), which
// column_sums_kernel adds in block order.  Bound by reading dz (134 MB a branch
// at batch 256) and by the 160 fp32 sums a pixel feeds, two to an fma.f32x2: a
// thread keeps the 80 of eight channels in registers over all its pixels, four
// neighbours at a time.  36 us for both branches at batch 64 (as im2col,
// transposes and a GEMM: about 400 us).
constexpr int kW0Sums = 10 * kConv0Out, kW0Blocks = 152;  // blocks of a branch: two an SM
__global__ void __launch_bounds__(256, 2) conv0_wgrad_kernel(const GradPair p, int H, int lwo4, uint32_t quads,
                                                             float *__restrict__ part) {
    __shared__ float red[8][kW0Sums];
    const bool br = blockIdx.y;
    const __nv_bfloat16 *img0 = br ? p.x[1] : p.x[0];
    const uint4 *dz = reinterpret_cast<const uint4 *>(br ? p.dz[1] : p.dz[0]);
    const int half = threadIdx.x & 1, Ho = H / 2;
    unsigned long long acc[10][4];
#pragma unroll
    for (int k = 0; k < 10; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = 0ull;
#pragma unroll 1
    for (uint32_t g = (blockIdx.x * 256 + threadIdx.x) >> 1; g < quads; g += gridDim.x * 128) {  // pixels 4g .. 4g + 3
        const int wq = (int)(g & ((1u << lwo4) - 1)), ho = (int)((g >> lwo4) % (uint32_t)Ho);
        const __nv_bfloat16 *img = img0 + (size_t)((g >> lwo4) / (uint32_t)Ho) * H * H;
        unsigned long long d[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 v = __ldg(dz + ((size_t)g * 4 + q) * 2 + half);
            const uint32_t vs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // bf16 = the upper half of an fp32
                d[q][j] = pack2(__uint_as_float(vs[j] << 16), __uint_as_float(vs[j] & 0xFFFF0000u));
                add2(acc[9][j], d[q][j]);
            }
        }
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
            const int h = 2 * ho - 1 + ky;  // < H: only the row above the image is missing
            if (h < 0) continue;
            const __nv_bfloat16 *row = img + (size_t)h * H + 8 * wq;  // columns 8 wq - 1 .. 8 wq + 7
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(row));
            const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
            float v[9];
            v[0] = wq > 0 ? __bfloat162float(row[-1]) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                v[2 * i + 1] = __uint_as_float(xs[i] << 16);
                v[2 * i + 2] = __uint_as_float(xs[i] & 0xFFFF0000u);
            }
#pragma unroll
            for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned long long vv = pack2(v[2 * q + kx], v[2 * q + kx]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) fma2(acc[3 * ky + kx][j], vv, d[q][j]);
                }
        }
    }
    // Over the lanes of equal half, then over the warps.
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 10; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 a = unpack2(acc[k][j]);
#pragma unroll
            for (int o = 16; o > 1; o >>= 1) {
                a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
                a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
            }
            if (lane < 2) *reinterpret_cast<float2 *>(&red[threadIdx.x >> 5][k * kConv0Out + 8 * half + 2 * j]) = a;
        }
    __syncthreads();
    if (threadIdx.x < kW0Sums) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
        part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kW0Sums + threadIdx.x] = t;
    }
}

// Average pooling and linear head of both branches (blockIdx.y), one CTA of
// 256 threads (one per channel) per example.
__global__ void __launch_bounds__(256) pool_head_kernel(const HeadPair p, int HW) {
    constexpr int C = 256;
    __shared__ float warp_sum[C / 32];
    const int n = blockIdx.x, c = threadIdx.x;
    const bool br = blockIdx.y;
    const __nv_bfloat16 *y = (br ? p.y[1] : p.y[0]) + (size_t)n * HW * C + c;
    float s = 0.f;
#pragma unroll 8
    for (int i = 0; i < HW; ++i) s += __bfloat162float(y[(size_t)i * C]);
    s /= (float)HW;
    (br ? p.feat[1] : p.feat[0])[(size_t)n * C + c] = s;
    float d = s * (br ? p.w[1] : p.w[0])[c];
#pragma unroll
    for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if ((c & 31) == 0) warp_sum[c >> 5] = d;
    __syncthreads();
    if (c == 0) {
        float t = 0.f;
        for (int w = 0; w < C / 32; ++w) t += warp_sum[w];
        (br ? p.logit[1] : p.logit[0])[n] = t + (br ? p.b[1] : p.b[0])[0];
    }
}

__device__ __forceinline__ float sigmoidf(float x) { return 1.f / (1.f + expf(-x)); }

// Fused probability p = s1 * s2 (s = sigmoid of each branch's logit) and,
// with labels, the binary cross-entropy of p and its derivative with
// respect to both logits (mean over the batch).
__global__ void fuse_loss_kernel(const float *__restrict__ l1, const float *__restrict__ l2,
                                 const float *__restrict__ label, int Nb, float *__restrict__ prob,
                                 float *__restrict__ dl1, float *__restrict__ dl2, float *__restrict__ loss) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= Nb) return;
    const float s1 = sigmoidf(l1[n]), s2 = sigmoidf(l2[n]);
    const float p = s1 * s2;
    if (prob) prob[n] = p;
    if (!label) return;
    const float y = label[n];
    const float pc = fminf(fmaxf(p, 1e-7f), 1.f - 1e-7f);
    atomicAdd(loss, -(y * logf(pc) + (1.f - y) * logf(1.f - pc)) / (float)Nb);
    // dL/dp = (p - y) / (p (1 - p)); dp/dl1 = p (1 - s1); dp/dl2 = p (1 - s2).
    const float g = (pc - y) / (1.f - pc) / (float)Nb;
    dl1[n] = g * (1.f - s1);
    dl2[n] = g * (1.f - s2);
}

// Head, pooling and last ReLU backward of both branches (blockIdx.y; C = 256
// channels).  Blocks 0 .. 7: dw[c] += sum_n dl[n] feat[n][c] of 32 channels, and
// db += sum_n dl[n] (block 0); block 8 + n: example n's
// dz[n][i][c] = dl[n] w[c] / HW where y > 0.
constexpr int kHeadBlocks = 8;
__global__ void __launch_bounds__(256) head_back_kernel(const HeadGrad p, int Nb, int HW) {
    constexpr int C = 256;
    __shared__ float red[8][32];
    const bool br = blockIdx.y;
    const float *dl = br ? p.dl[1] : p.dl[0];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (blockIdx.x < kHeadBlocks) {
        const int c = blockIdx.x * 32 + lane;
        const float *feat = br ? p.feat[1] : p.feat[0];
        float s = 0.f;
#pragma unroll 8
        for (int n = warp; n < Nb; n += 8) s += dl[n] * feat[n * C + c];
        red[warp][lane] = s;
        __syncthreads();
        if (warp == 0) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) t += red[w][lane];
            (br ? p.dw[1] : p.dw[0])[c] += t;
        } else if (warp == 1 && blockIdx.x == 0) {
            float t = 0.f;
            for (int n = lane; n < Nb; n += 32) t += dl[n];
#pragma unroll
            for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) (br ? p.db[1] : p.db[0])[0] += t;
        }
        return;
    }
    const int n = blockIdx.x - kHeadBlocks;
    const float *w = (br ? p.w[1] : p.w[0]) + 8 * lane;
    uint32_t g[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) g[e] = __bfloat16_as_ushort(__float2bfloat16(dl[n] * w[e] / (float)HW));
    const size_t at = (size_t)n * HW * (C / 8) + lane;
    const uint4 *y = reinterpret_cast<const uint4 *>(br ? p.y[1] : p.y[0]) + at;
    uint4 *dz = reinterpret_cast<uint4 *>(br ? p.dz[1] : p.dz[0]) + at;
#pragma unroll 4
    for (int i = warp; i < HW; i += 8) {
        const uint4 v = y[(size_t)i * (C / 8)];
        const uint32_t vs[4] = {v.x, v.y, v.z, v.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            o[e] = (__uint_as_float(vs[e] << 16) > 0.f ? g[2 * e] : 0u) |
                   (__uint_as_float(vs[e] & 0xFFFF0000u) > 0.f ? g[2 * e + 1] << 16 : 0u);
        dz[(size_t)i * (C / 8)] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// Bias gradients, the sums of dz[p][c] over the pixels, in two deterministic
// stages.  Here chunk blockIdx.x of the P rows of both branches (blockIdx.y) to
// part[branch][chunk][c]: a thread adds eight channels (16 bytes) of every
// (2048 / C)-th row, then the block's threads of equal channels form a tree.  Bound
// by reading dz; all layers of both branches at batch 64, both stages: 415 us with
// 2-byte loads and a serial second stage -> 38 us.
__global__ void __launch_bounds__(256, 4) bias_part_kernel(const __nv_bfloat16 *__restrict__ dz0,
                                                        const __nv_bfloat16 *__restrict__ dz1, int64_t P, int C,
                                                        int64_t rows_per_chunk, float *__restrict__ part) {
    __shared__ float red[8][256];
    const int c8 = C / 8, lanes = 256 / c8, row = threadIdx.x / c8, col = threadIdx.x - row * c8;
    const uint4 *dz = reinterpret_cast<const uint4 *>(blockIdx.y ? dz1 : dz0) + col;
    const int64_t p1 = min(P, (blockIdx.x + 1) * rows_per_chunk);
    float a[8] = {};
#pragma unroll 4
    for (int64_t p = blockIdx.x * rows_per_chunk + row; p < p1; p += lanes) {
        const uint4 v = __ldg(dz + p * c8);
        const uint32_t vs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            a[2 * e] += __uint_as_float(vs[e] << 16);
            a[2 * e + 1] += __uint_as_float(vs[e] & 0xFFFF0000u);
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) red[e][threadIdx.x] = a[e];
    for (int s = lanes / 2; s; s >>= 1) {
        __syncthreads();
        if (row < s)
#pragma unroll
            for (int e = 0; e < 8; ++e) red[e][threadIdx.x] += red[e][threadIdx.x + s * c8];
    }
    // the first c8 threads hold the sums (each its own: no barrier needed)
    if (row == 0)
#pragma unroll
        for (int e = 0; e < 8; ++e)
            part[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * C + 8 * col + e] = red[e][threadIdx.x];
}

// The second stage for every layer (blockIdx.z) of both branches (blockIdx.y):
// 32 columns a block; warp w adds rows w, w + 32, ... in order, then the warps' sums
// are added in order.  Layer 0's columns are its weight gradients' and biases'.
__global__ void __launch_bounds__(1024) column_sums_kernel(const ColumnSums p) {
    __shared__ float red[32][33];
    const int l = blockIdx.z, cols = p.cols[l], n = p.rows[l];
    const int c = blockIdx.x * 32 + threadIdx.x, w = threadIdx.y;
    if ((int)blockIdx.x * 32 >= cols) return;
    float s = 0.f;
    if (c < cols) {
        const float *q = p.part[l] + (size_t)blockIdx.y * n * cols + c;
#pragma unroll 4
        for (int r = w; r < n; r += 32) s += q[(size_t)r * cols];
    }
    red[w][threadIdx.x] = s;
    __syncthreads();
    if (w || c >= cols) return;
    float t = 0.f;
#pragma unroll
    for (int r = 0; r < 32; ++r) t += red[r][threadIdx.x];
    float *db = blockIdx.y ? p.db[1][l] : p.db[0][l];
    if (l > 0) db[c] += t;
    else if (c < 9 * kConv0Out) (blockIdx.y ? p.dw0[1] : p.dw0[0])[(c & 15) * p.kp0 + (c >> 4)] += t;
    else db[c - 9 * kConv0Out] += t;
}

// Adam on fp32 master weights; bf16 copy refreshed for the GEMMs.
__global__ void adam_kernel(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2, __nv_bfloat16 *__restrict__ wb) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        if (wb) wb[i] = __float2bfloat16(wi);
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ a, int64_t n, __nv_bfloat16 *__restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16(a[i]);
}

__global__ void to_flat_kernel(const FlatLayout f, const float *__restrict__ b0, const float *__restrict__ b1,
                               int64_t count, float *__restrict__ out) {
    const float *src = blockIdx.y ? b1 : b0;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int e = i, s = 0;
    while (s < f.segments && e >= f.rows[s] * f.cols[s]) {
        e -= f.rows[s] * f.cols[s];
        ++s;
    }
    if (s < f.segments) out[blockIdx.y * count + i] = src[f.off[s] + (int64_t)(e / f.cols[s]) * f.ld[s] + e % f.cols[s]];
}

// Images of one candidate from its subband dynamic spectrum sub[S][T_in]
// (already dedispersed at the candidate DM within each subband; time bins):
//   ft[s][u]  = sub[s][u0 + u]                         (S x 256)
//   dmt[j][u] = sum_s sub[s][u0 + u + shift[j][s]]     (256 trial-DM offsets)
// u0 = (T_in - 256) / 2, bins outside the spectrum count 0, subbands added in
// order.  Each image is then set to zero mean and unit variance (computed in
// fp32 over its 65536 values) and stored as bf16.
//
// DM-time rows: one CTA per (32 rows j, candidate), one warp per R rows of
// 256 bins (a lane's bins are lane + 32 i).  The sum is bound by shared-memory
// reads and instruction issue.  Neighbouring rows read most subbands at the
// same shift (the shifts of a 255-bin sweep differ by at most one bin from
// row to row, at the band's bottom), so a warp keeps the bins it has loaded
// and loads again only where the shift changes: about 0.4 loads per row and
// subband; one address serves a lane's eight bins, and two bins are added per
// instruction (add.f32x2, the same rounding as two adds).  Windows of
// [smallest, largest shift of the 32 rows] + 256 bins arrive by 16-byte
// asynchronous copies, several subbands to a stage, two stages.  The shifts
// are any integers: wide ones take fewer subbands per stage, and where not even
// one window fits a stage the bins are read from global memory.
// 512-bin spectra: 1.00 -> 0.35 ms at batch 256 and 0.175 -> 0.046 ms at batch 5
// against one load, one address and one add per bin and row.
constexpr int kFeatRows = 32;
constexpr int kFeatStage = 8 * 336;  // floats of one stage

template <int R>
__global__ void __launch_bounds__(32 * kFeatRows / R) features_raw_kernel(const float *__restrict__ sub, int T_in,
                                                                        const int32_t *__restrict__ shift, bool vec,
                                                                        float *dmt_raw,
                                                                        float4 *__restrict__ part) {
    constexpr int NW = kFeatRows / R, NT = 32 * NW, NI = kImg / 32;
    __shared__ __align__(16) float win[2][kFeatStage];
    __shared__ __align__(16) uint16_t rel[kImg][kFeatRows];  // bin of a row's u = 0 in its subband's window
    __shared__ int base[kImg];                               // first bin of the window (a multiple of 4)
    __shared__ float2 col_sum[2][NI];
    __shared__ int widest;
    const int b = blockIdx.y, j0 = blockIdx.x * kFeatRows, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = (T_in - kImg) / 2;
    const float *sb = sub + (size_t)b * kImg * T_in;
    if (threadIdx.x == 0) widest = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < kImg; k += NT) {
        // A shift that leaves the spectrum altogether reads zeros only: clamped to the first that does.
        auto at = [&](int r) { return u0 + min(max(shift[(size_t)(j0 + r) * kImg + k], -u0 - kImg), T_in - u0); };
        int lo = at(0), hi = lo;
        for (int r = 1; r < kFeatRows; ++r) {
            const int v = at(r);
            lo = min(lo, v);
            hi = max(hi, v);
        }
        lo &= ~3;
        base[k] = lo;
        for (int r = 0; r < kFeatRows; ++r) rel[k][r] = (uint16_t)(at(r) - lo);
        atomicMax(&widest, hi - lo);
    }
    __syncthreads();
    const int stride = (kImg + widest + 3) & ~3;        // floats of a window
    const int per = min(8, kFeatStage / stride);        // subbands of a stage (0: straight from global memory)
    auto stage = [&](int k0, int buf) {
        for (int kk = warp; kk < per && k0 + kk < kImg; kk += NW) {
            const int e0 = base[k0 + kk];
            const float *src = sb + (size_t)(k0 + kk) * T_in;
            float *dst = &win[buf][kk * stride];
            if (vec) {  // rows start at 16-byte boundaries: a group of four bins is inside or outside as one
                for (int c = 4 * lane; c < stride; c += 128) {
                    const bool ok = e0 + c >= 0 && e0 + c < T_in;
                    cp_async16(dst + c, src + (ok ? e0 + c : 0), ok);
                }
            } else {
                for (int c = lane; c < stride; c += 32) {
                    if (e0 + c >= 0 && e0 + c < T_in) cp_async4(dst + c, src + e0 + c);
                    else dst[c] = 0.f;
                }
            }
        }
        cp_async_commit();
    };
    unsigned long long acc[R][NI / 2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < NI / 2; ++i) acc[r][i] = 0ull;
    unsigned long long v[NI / 2];
    auto rows_of = [&](int k, uint32_t (&o)[R]) {
        const uint16_t *p = &rel[k][warp * R];
        if constexpr (R == 8) {
            const uint4 w = *reinterpret_cast<const uint4 *>(p);
            const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int r = 0; r < 8; ++r) o[r] = (x[r >> 1] >> (16 * (r & 1))) & 0xFFFFu;
        } else if constexpr (R == 4) {
            const uint2 w = *reinterpret_cast<const uint2 *>(p);
            o[0] = w.x & 0xFFFFu, o[1] = w.x >> 16, o[2] = w.y & 0xFFFFu, o[3] = w.y >> 16;
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) o[r] = p[r];
        }
    };
    if (per > 0) {
        stage(0, 0);
        for (int k0 = 0, buf = 0; k0 < kImg; k0 += per, buf ^= 1) {
            stage(k0 + per, buf ^ 1);
            cp_async_wait<1>();
            __syncthreads();
            const int nk = min(per, kImg - k0);
            for (int kk = 0; kk < nk; ++kk) {
                const float *p = &win[buf][kk * stride + lane];
                uint32_t o[R];
                rows_of(k0 + kk, o);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (r == 0 || o[r] != o[r - 1]) {
#pragma unroll
                        for (int i = 0; i < NI / 2; ++i) v[i] = pack2(p[o[r] + 64 * i], p[o[r] + 64 * i + 32]);
                    }
#pragma unroll
                    for (int i = 0; i < NI / 2; ++i) add2(acc[r][i], v[i]);
                }
            }
            __syncthreads();
        }
    } else {
        for (int k = 0; k < kImg; ++k) {
            uint32_t o[R];
            rows_of(k, o);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int e = base[k] + (int)o[r] + lane;
                auto bin = [&](int i) {
                    const int x = e + 32 * i;
                    return x >= 0 && x < T_in ? __ldg(sb + (size_t)k * T_in + x) : 0.f;
                };
#pragma unroll
                for (int i = 0; i < NI / 2; ++i) add2(acc[r][i], pack2(bin(2 * i), bin(2 * i + 1)));
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float2 d2 = unpack2(acc[r][i >> 1]);
            dmt_raw[((size_t)b * kImg + j0 + warp * R + r) * kImg + 32 * i + lane] = i & 1 ? d2.y : d2.x;
        }
    __syncthreads();
    // The block's sums of both images: each column's rows in order, a warp tree
    // over 32 columns, then those in turn, whatever R is (the normalisation adds
    // the blocks in turn).  The variance is a small difference of large sums, so
    // this order is part of the result.
    for (int it = warp; it < 2 * NI; it += NW) {
        const int img = it / NI, u = (it % NI) * 32 + lane;
        const float *col = img ? dmt_raw + ((size_t)b * kImg + j0) * kImg + u : sb + (size_t)j0 * T_in + u0 + u;
        const int row = img ? kImg : T_in;
        float t = 0.f, t2 = 0.f;
#pragma unroll 16
        for (int r = 0; r < kFeatRows; ++r) {
            const float v = col[(size_t)r * row];
            t += v;
            t2 += v * v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t += __shfl_xor_sync(0xffffffffu, t, o);
            t2 += __shfl_xor_sync(0xffffffffu, t2, o);
        }
        if (lane == 0) col_sum[img][it % NI] = make_float2(t, t2);
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float2 a = col_sum[threadIdx.x][0];
        for (int w = 1; w < NI; ++w) {
            a.x += col_sum[threadIdx.x][w].x;
            a.y += col_sum[threadIdx.x][w].y;
        }
        reinterpret_cast<float2 *>(part + (size_t)b * (kImg / kFeatRows) + blockIdx.x)[threadIdx.x] = a;
    }
}

// One CTA per (block of kFeatRows rows, candidate, image): the image's mean
// and population variance from the feature kernel's per-block sums (added
// in block order), then the block's rows scaled and stored as bf16.  The
// frequency-time rows come straight from the spectrum.
__global__ void __launch_bounds__(kImg) normalise_kernel(const float *__restrict__ sub, int T_in,
                                                         const float *__restrict__ dmt_raw,
                                                         const float4 *__restrict__ part, __nv_bfloat16 *__restrict__ ft,
                                                         __nv_bfloat16 *__restrict__ dmt) {
    const int b = blockIdx.y, img = blockIdx.z, j0 = blockIdx.x * kFeatRows, u = threadIdx.x;
    float s = 0.f, s2 = 0.f;
    for (int q = 0; q < kImg / kFeatRows; ++q) {
        const float4 p = part[(size_t)b * (kImg / kFeatRows) + q];
        s += img ? p.z : p.x;
        s2 += img ? p.w : p.y;
    }
    const float n = (float)(kImg * kImg);
    const float mean = s / n;
    const float var = fmaxf(s2 / n - mean * mean, 0.f);
    const float inv = var > 0.f ? rsqrtf(var) : 0.f;
    const float *raw = img ? dmt_raw + (size_t)b * kImg * kImg : sub + (size_t)b * kImg * T_in + (T_in - kImg) / 2;
    const int row = img ? kImg : T_in;
    __nv_bfloat16 *out = (img ? dmt : ft) + (size_t)b * kImg * kImg;
#pragma unroll 8
    for (int r = 0; r < kFeatRows; ++r)
        out[(j0 + r) * kImg + u] = __float2bfloat16((raw[(size_t)(j0 + r) * row + u] - mean) * inv);
}

// Subband dynamic spectrum of candidate q from the staged beam xt
// [nchan][pitch]: sub[q][s][u] = sum over the channels c of subband s and
// i < dec of xt[c][t0 + (u - t_in/2) * dec + i + delay[dm][c]], with t0 the
// centre of the candidate's boxcar window; samples outside [0, n_in) count 0.
// One CTA per (candidate, subband), threads over time bins; the sums are
// integers, so their order is free.  Bound by instruction issue on addresses and bounds
// and, for bins of many samples, by loads whose lanes lie far apart: a window that
// lies inside the beam in every channel of the subband is read without checks
// from one address and offsets the CTA shares, and bins of eight samples or more four
// samples at a time (the ends of a bin masked) where rows are 4-byte aligned.  Windows
// that leave the beam (all of a wide candidate's in a short gulp) clamp each bin and
// are read the same way.  4096 channels, 512 bins, one load, check and add per sample
// against this: 60 candidates of width 1 inside the beam 200 -> 43 us, at its edge
// 194 -> 151; five of width 64 at the edge 76 -> 42, of width 256 644 -> 265.
// The widths are read in the parameters' own memory: a copy of them on the stack, which
// an index makes, costs 25 us of launches of 15360 CTAs.
constexpr int kExtractPer = 256;  // channels of a subband that share offsets

// A subband of a window that leaves the beam, or of too many channels to share
// offsets: every channel's samples inside the beam.
__device__ __forceinline__ void extract_edge(const uint8_t *__restrict__ rows, int64_t pitch, int64_t n_in,
                                          const int32_t *__restrict__ dl, int per, int64_t first, int dec, int t_in,
                                          bool words, float *__restrict__ out) {
    for (int u = threadIdx.x; u < t_in; u += 256) {
        const int64_t tb = first + (int64_t)u * dec;
        uint32_t acc = 0;
        if (dec < 4) {
#pragma unroll 4
            for (int k = 0; k < per; ++k) {
                const int64_t t = tb + __ldg(dl + k);
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    if (i < dec && t + i >= 0 && t + i < n_in) acc += __ldg(rows + k * pitch + t + i);
            }
        } else if (dec < 8 || !words) {
            for (int k = 0; k < per; ++k) {
                const int64_t t = tb + __ldg(dl + k), lo = max(t, (int64_t)0), hi = min(t + dec, n_in);
                const uint8_t *r = rows + k * pitch;
#pragma unroll 4
                for (int64_t i = lo; i < hi; ++i) acc += __ldg(r + i);
            }
        } else {
#pragma unroll 2
            for (int k = 0; k < per; ++k) {
                const int64_t t = tb + __ldg(dl + k), lo = max(t, (int64_t)0), hi = min(t + dec, n_in);
                if (lo >= hi) continue;
                const uint8_t *r = rows + k * pitch + lo;
                const int skip = (int)(reinterpret_cast<uintptr_t>(r) & 3), end = skip + (int)(hi - lo) - 1;
                const uint32_t *w = reinterpret_cast<const uint32_t *>(r - skip);
                const int last = end >> 2;
                const uint32_t tail = 0xFFFFFFFFu >> (8 * (3 - (end & 3)));
                acc = __dp4a((__ldg(w) & (last ? 0xFFFFFFFFu : tail)) >> (8 * skip), 0x01010101u, acc);
#pragma unroll 4
                for (int i = 1; i < last; ++i) acc = __dp4a(__ldg(w + i), 0x01010101u, acc);
                if (last) acc = __dp4a(__ldg(w + last) & tail, 0x01010101u, acc);
            }
        }
        out[u] = (float)acc;
    }
}

__global__ void __launch_bounds__(256) extract_kernel(const uint8_t *__restrict__ xt, int64_t pitch, int64_t n_in,
                                                      int32_t nchan, const int32_t *__restrict__ delays,
                                                      const sp_cand *__restrict__ cands,
                                                      const __grid_constant__ ExtractWidths wt, int32_t nsub,
                                                      int32_t t_in, bool words, float *__restrict__ sub) {
    __shared__ int64_t off_s[kExtractPer];
    const int q = blockIdx.y, s = blockIdx.x;
    const sp_cand c = cands[q];
    const int per = nchan / nsub;
    const int wi = min(max(c.width_idx, 0), SP_MAX_WIDTHS - 1);
    const int dec = wt.dec[wi];
    const int64_t first = (int64_t)c.t + wt.half[wi] - (int64_t)(t_in / 2) * dec;  // sample of bin 0 without delay
    const int32_t *dl = delays + (int64_t)c.dm_idx * nchan + s * per;
    const uint8_t *rows = xt + (int64_t)s * per * pitch;
    float *out = sub + ((int64_t)q * nsub + s) * t_in;
    bool inside = per <= kExtractPer;
    if (inside && (int)threadIdx.x < per) {
        const int64_t d = dl[threadIdx.x];
        inside = first + d >= 0 && first + d + (int64_t)t_in * dec <= n_in;
        off_s[threadIdx.x] = threadIdx.x * pitch + d;
    }
    if (__syncthreads_and(inside)) {
        for (int u = threadIdx.x; u < t_in; u += 256) {
            const uint8_t *p = rows + first + (int64_t)u * dec;
            uint32_t acc = 0;
            if (dec == 1) {
#pragma unroll 8
                for (int k = 0; k < per; ++k) acc += __ldg(p + off_s[k]);
            } else if (dec < 8 || !words) {
#pragma unroll 4
                for (int k = 0; k < per; ++k) {
                    const uint8_t *r = p + off_s[k];
#pragma unroll 4
                    for (int i = 0; i < dec; ++i) acc += __ldg(r + i);
                }
            } else {
#pragma unroll 2
                for (int k = 0; k < per; ++k) {
                    const uint8_t *r = p + off_s[k];
                    const int skip = (int)(reinterpret_cast<uintptr_t>(r) & 3);
                    const uint32_t *w = reinterpret_cast<const uint32_t *>(r - skip);
                    const int last = (skip + dec - 1) >> 2;  // >= 1; a word of the row, whose pitch is whole words
                    acc = __dp4a(__ldg(w) >> (8 * skip), 0x01010101u, acc);
#pragma unroll 4
                    for (int i = 1; i < last; ++i) acc = __dp4a(__ldg(w + i), 0x01010101u, acc);
                    acc = __dp4a(__ldg(w + last) & (0xFFFFFFFFu >> (8 * (3 - ((skip + dec - 1) & 3)))), 0x01010101u, acc);
                }
            }
            out[u] = (float)acc;
        }
        return;
    }
    extract_edge(rows, pitch, n_in, dl, per, first, dec, t_in, words, out);
}

int grid_for(int64_t n, int threads = 256) {
    return (int)std::min<int64_t>((n + threads - 1) / threads, 152 * 32);
}

}  // namespace

int cnn_conv0(const ConvPair &p, int Nb, int H, int Kp, cudaStream_t st) {
    const int Ho = H / 2;
    const int64_t P = (int64_t)Nb * Ho * Ho;
    uintptr_t all = 0;
    for (int b = 0; b < 2; ++b) all |= reinterpret_cast<uintptr_t>(p.x[b]) | reinterpret_cast<uintptr_t>(p.y[b]);
    int lwo4 = 0;
    while ((4 << lwo4) < Ho) ++lwo4;
    if (P >= ((int64_t)1 << 31) || Kp < 9 || (all & 15) || (4 << lwo4) != Ho) return SP_ELIMIT;
    const uint32_t quads = (uint32_t)(P / 4);
    conv0_kernel<<<dim3((quads + 255) / 256, 2), 256, 0, st>>>(p, H, lwo4, quads, Kp);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_conv0_wgrad(const GradPair &p, int Nb, int H, float *part, int *rows, cudaStream_t st) {
    const uint32_t quads = (uint32_t)((int64_t)Nb * (H / 2) * (H / 2) / 4);
    int lwo4 = 0;
    while ((8 << lwo4) < H) ++lwo4;
    *rows = (int)std::min<uint32_t>(kW0Blocks, (quads + 127) / 128);
    conv0_wgrad_kernel<<<dim3((unsigned)*rows, 2), 256, 0, st>>>(p, H, lwo4, quads, part);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_bias_part(const GradPair &p, int64_t P, int C, float *part, int *rows, cudaStream_t st) {
    if (C < 16 || C > 256 || 256 % C || P < 1) return SP_EINVAL;
    const int64_t chunks = std::min<int64_t>(kBiasChunks, (P + 255) / 256), per = (P + chunks - 1) / chunks;
    *rows = (int)((P + per - 1) / per);
    bias_part_kernel<<<dim3((unsigned)*rows, 2), 256, 0, st>>>(p.dz[0], p.dz[1], P, C, per, part);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_column_sums(const ColumnSums &p, cudaStream_t st) {
    int most = 0;
    for (int l = 0; l < kCnnLayers; ++l) most = std::max(most, p.cols[l]);
    column_sums_kernel<<<dim3((unsigned)((most + 31) / 32), 2, kCnnLayers), dim3(32, 32), 0, st>>>(p);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_pool_head(const HeadPair &p, int Nb, int HW, cudaStream_t st) {
    pool_head_kernel<<<dim3((unsigned)Nb, 2), 256, 0, st>>>(p, HW);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_fuse_loss(const float *l1, const float *l2, const float *label, int Nb, float *prob, float *dl1, float *dl2,
                  float *loss, cudaStream_t st) {
    fuse_loss_kernel<<<(Nb + 255) / 256, 256, 0, st>>>(l1, l2, label, Nb, prob, dl1, dl2, loss);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_head_back(const HeadGrad &p, int Nb, int HW, cudaStream_t st) {
    head_back_kernel<<<dim3((unsigned)(kHeadBlocks + Nb), 2), 256, 0, st>>>(p, Nb, HW);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_adam(float *w, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2, float eps,
             int64_t step, __nv_bfloat16 *wb, cudaStream_t st) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    adam_kernel<<<grid_for(n), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2, wb);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_to_flat(const FlatLayout &f, const float *b0, const float *b1, int64_t count, float *out, cudaStream_t st) {
    to_flat_kernel<<<dim3((unsigned)((count + 255) / 256), 2), 256, 0, st>>>(f, b0, b1, count, out);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_to_bf16(const float *a, int64_t n, __nv_bfloat16 *b, cudaStream_t st) {
    to_bf16_kernel<<<grid_for(n), 256, 0, st>>>(a, n, b);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_extract(const uint8_t *xt, int64_t pitch, int64_t n_in, int32_t nchan, const int32_t *delays,
                const sp_cand *cands, int32_t ncand, const ExtractWidths &wt, int32_t nsub, int32_t t_in, float *sub,
                cudaStream_t st) {
    const bool words = ((reinterpret_cast<uintptr_t>(xt) | (uintptr_t)pitch) & 3) == 0;
    extract_kernel<<<dim3((unsigned)nsub, (unsigned)ncand), 256, 0, st>>>(xt, pitch, n_in, nchan, delays, cands, wt,
                                                                        nsub, t_in, words, sub);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int cnn_features(const float *sub, int Nb, int S, int T_in, const int32_t *shift, float *dmt_raw, float *part,
                 __nv_bfloat16 *ft, __nv_bfloat16 *dmt, cudaStream_t st) {
    if (S != kImg || T_in < kImg || T_in > 4096) return SP_EINVAL;
    float4 *p4 = reinterpret_cast<float4 *>(part);
    const bool vec = T_in % 4 == 0 && (reinterpret_cast<uintptr_t>(sub) & 15) == 0;
    // Rows per warp: more share more loads, fewer give more warps.
    const dim3 grid(kImg / kFeatRows, Nb);
    if (Nb >= 48) features_raw_kernel<8><<<grid, 32 * kFeatRows / 8, 0, st>>>(sub, T_in, shift, vec, dmt_raw, p4);
    else if (Nb >= 16) features_raw_kernel<4><<<grid, 32 * kFeatRows / 4, 0, st>>>(sub, T_in, shift, vec, dmt_raw, p4);
    else features_raw_kernel<2><<<grid, 32 * kFeatRows / 2, 0, st>>>(sub, T_in, shift, vec, dmt_raw, p4);
    note_launch();
    if (cudaGetLastError() != cudaSuccess) return SP_ECUDA;
    normalise_kernel<<<dim3(kImg / kFeatRows, Nb, 2), kImg, 0, st>>>(sub, T_in, dmt_raw, p4, ft, dmt);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

}  // namespace sp
