// sp_cnn_internal.h -- declarations shared by the classifier's kernels
// (cnn.cu) and its host orchestration (cnn.cpp).  Not installed.
#pragma once

#include <cuda_bf16.h>

#include "sp_internal.h"

namespace sp {

constexpr int kImg = 256;  // images are kImg x kImg (subbands or trial DMs x time bins)
constexpr int kCnnLayers = 5;

// The two branches' operands of a layer.
struct ConvPair {
    const __nv_bfloat16 *x[2], *w[2];
    const float *bias[2];
    __nv_bfloat16 *y[2];
};
// The layers 1 to 4 of both branches on the tensor cores (cnn_tc.cu): 3x3,
// stride 2, zero padding 1, from C to 2 C channels.  x NHWC bf16 [Nb][H][H][C], w
// [2 C][Kp] bf16 (k = tap*C + c; Kp >= 9 C, a multiple of 8), y and dz
// [Nb*(H/2)^2][2 C] bf16, all 16-byte aligned; C 16..128, H 128..16, powers of two.
// y = relu(conv(x) + bias).
// A wait of theirs that runs out sets *status (host-visible) to SP_STATUS_STAGING_TIMEOUT.
int cnn_conv_fwd(const ConvPair &p, int Nb, int H, int C, int Kp, int32_t *status, cudaStream_t st);
// Operands of a layer's gradients: input x, dz (of the layer's output before its
// ReLU), weights; dx is the dz of the layer below, dw fp32 [2 C][Kp].
struct GradPair {
    const __nv_bfloat16 *x[2], *dz[2], *w[2];
    __nv_bfloat16 *dx[2];
    float *dw[2];
};
// dw += dz^T x (part: cnn_wgrad_part_floats of at least Nb, workspace; the split
// over pixels and the order of its sums depend on the shape only).
int64_t cnn_wgrad_part_floats(int Nb, int H, int C, int Kp);
int cnn_conv_wgrad(const GradPair &p, int Nb, int H, int C, int Kp, float *part, int32_t *status, cudaStream_t st);
// dx = (transposed convolution of dz) where x > 0, else 0 (x and dx 32-byte aligned).
int cnn_conv_dgrad(const GradPair &p, int Nb, int H, int C, int Kp, int32_t *status, cudaStream_t st);
// Layer 0 of both branches (one input channel, 16 outputs, 3x3, stride 2,
// padding 1) as a direct convolution with bias and ReLU: x [Nb][H][H] (H a
// multiple of 8), y [Nb*(H/2)^2][16] bf16, both 16-byte aligned, weights w
// [16][Kp] bf16 (taps 0..8 used), bias [16] fp32.
int cnn_conv0(const ConvPair &p, int Nb, int H, int Kp, cudaStream_t st);
// Sums of its weight and bias gradients: part[2][*rows][160] (at most kBiasChunks
// rows), columns tap * 16 + co, then the biases.
constexpr int kBiasChunks = 512;
int cnn_conv0_wgrad(const GradPair &p, int Nb, int H, float *part, int *rows, cudaStream_t st);
// Sums of dz's P rows: part[2][*rows][C] (C 16..256, a power of two; at most kBiasChunks rows).
int cnn_bias_part(const GradPair &p, int64_t P, int C, float *part, int *rows, cudaStream_t st);
// Adds the rows of every layer's part (cols columns; layer 0 as cnn_conv0_wgrad
// leaves it) to the bias gradients db and layer 0's weight gradients dw0 [16][kp0].
struct ColumnSums {
    const float *part[kCnnLayers];
    int rows[kCnnLayers], cols[kCnnLayers];
    float *db[2][kCnnLayers], *dw0[2];
    int kp0;
};
int cnn_column_sums(const ColumnSums &p, cudaStream_t st);
// Average pooling and linear head of both branches (C = 256 channels):
// feat[n][c] = mean over HW of y, logit[n] = feat[n] . w + b[0].
struct HeadPair {
    const __nv_bfloat16 *y[2];
    const float *w[2], *b[2];
    float *feat[2], *logit[2];
};
int cnn_pool_head(const HeadPair &p, int Nb, int HW, cudaStream_t st);
// Back through head, pooling and last ReLU: dw [256] and db [1] added to, dz written.
struct HeadGrad {
    const float *feat[2], *dl[2], *w[2];
    const __nv_bfloat16 *y[2];
    __nv_bfloat16 *dz[2];
    float *dw[2], *db[2];
};
int cnn_head_back(const HeadGrad &p, int Nb, int HW, cudaStream_t st);
int cnn_fuse_loss(const float *l1, const float *l2, const float *label, int Nb, float *prob, float *dl1, float *dl2,
                  float *loss, cudaStream_t st);
int cnn_adam(float *w, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2, float eps,
             int64_t step, __nv_bfloat16 *wb, cudaStream_t st);
// out[branch][0 .. count) = the branch's segments one after the other, rows x cols
// each from rows of ld at off.
struct FlatLayout {
    int segments;
    int64_t off[2 * kCnnLayers + 2];
    int rows[2 * kCnnLayers + 2], cols[2 * kCnnLayers + 2], ld[2 * kCnnLayers + 2];
};
int cnn_to_flat(const FlatLayout &f, const float *b0, const float *b1, int64_t count, float *out, cudaStream_t st);
int cnn_to_bf16(const float *a, int64_t n, __nv_bfloat16 *b, cudaStream_t st);
// Decimation and half width of each trial width, passed by value.
struct ExtractWidths {
    int32_t dec[SP_MAX_WIDTHS];
    int32_t half[SP_MAX_WIDTHS];
};
int cnn_extract(const uint8_t *xt, int64_t pitch, int64_t n_in, int32_t nchan, const int32_t *delays,
                const sp_cand *cands, int32_t ncand, const ExtractWidths &wt, int32_t nsub, int32_t t_in, float *sub,
                cudaStream_t st);
// part: Nb * 8 float4 of workspace (per-block image sums, 16-byte aligned).
int cnn_features(const float *sub, int Nb, int S, int T_in, const int32_t *shift, float *dmt_raw, float *part,
                 __nv_bfloat16 *ft, __nv_bfloat16 *dmt, cudaStream_t st);

}  // namespace sp
