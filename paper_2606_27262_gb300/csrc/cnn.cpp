// cnn.cpp -- the candidate classifier (arXiv 2606.27262, Sec. 3.2.2): two
// convolutional networks, one on the frequency-time image and one on the
// DM-time image of a candidate, fused multiplicatively into one
// probability; forward, backward and Adam on the GPU with the kernels of
// cnn.cu.  The paper runs FETCH's pretrained DenseNet121/Xception pair; its
// weights and training data are not available, so this network is small
// (about 0.79 M parameters) and trained here.
//
// Per branch: five 3x3 convolutions with stride 2 and padding 1
// (1->16->32->64->128->256 channels, 256x256 -> 8x8), each followed by
// ReLU; global average pooling; a linear head to one logit.  p = s(l_ft) *
// s(l_dmt) with s the logistic function; the loss is the binary
// cross-entropy of p.  Activations are bf16 in NHWC order; weights have an
// fp32 master copy (Adam) and a bf16 copy (GEMM operand).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <random>
#include <vector>

#include "sp_cnn_internal.h"

using namespace sp;

namespace {

constexpr int kLayers = kCnnLayers;
constexpr int kCin[kLayers] = {1, 16, 32, 64, 128};
constexpr int kCout[kLayers] = {16, 32, 64, 128, 256};
constexpr int kHin[kLayers] = {256, 128, 64, 32, 16};
constexpr int kFeat = 256;
static_assert(kCin[0] == 1 && kCout[0] == 16, "cnn_conv0 computes the one-channel, 16-output first layer");
constexpr int kAlign = 64;  // parameter segments start at multiples of 64 elements (16-byte aligned bf16)

constexpr int kp_of(int l) { return ((9 * kCin[l] + 31) / 32) * 32; }
constexpr int ho_of(int l) { return kHin[l] / 2; }
int64_t up(int64_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
int part_cols(int l) { return l == 0 ? 10 * kCout[0] : kCout[l]; }  // of cnn_conv0_wgrad, cnn_bias_part

struct Branch {
    int64_t off_w[kLayers] = {}, off_b[kLayers] = {}, off_hw = 0, off_hb = 0, n = 0;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *pb = nullptr;  // bf16 mirror of params (GEMM weights)
    __nv_bfloat16 *y[kLayers] = {}, *dz[kLayers] = {};
    float *feat = nullptr, *logit = nullptr, *dl = nullptr;
};

}  // namespace

struct sp_cnn {
    int device = 0;
    int32_t max_batch = 0;
    Branch br[2];
    float *prob = nullptr, *loss = nullptr;
    float *sums = nullptr;   // partial sums of layer 0's gradients and of every bias gradient
    float *wpart = nullptr;  // partial weight gradients of a layer
    float *flat = nullptr;  // parameters or gradients in the external order, on their way out
    std::mutex flat_lock;   // held while `flat` is filled and copied
    int32_t *status = nullptr;  // page-locked, set by the tensor-core kernels (a bounded wait ran out)
    int64_t step = 0;
    bool have_grads = false;
};

namespace {

int dalloc(void **p, int64_t bytes) {
    if (cudaMalloc(p, (size_t)std::max<int64_t>(bytes, 256)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return SP_ENOMEM;
    }
    return SP_OK;
}

void layout(Branch &b) {
    int64_t o = 0;
    for (int l = 0; l < kLayers; ++l) {
        b.off_w[l] = o;
        o = up(o + (int64_t)kCout[l] * kp_of(l));
        b.off_b[l] = o;
        o = up(o + kCout[l]);
    }
    b.off_hw = o;
    o = up(o + kFeat);
    b.off_hb = o;
    b.n = up(o + 1);
}

// Flat external order per branch: for each layer W [Cout][9 Cin] then
// b [Cout]; then the head w [256] and b; branch 0 (frequency-time) first.
int64_t flat_count() {
    int64_t n = 0;
    for (int l = 0; l < kLayers; ++l) n += (int64_t)kCout[l] * 9 * kCin[l] + kCout[l];
    return n + kFeat + 1;
}

void from_flat(const Branch &b, const float *in, std::vector<float> &dev) {
    dev.assign((size_t)b.n, 0.f);
    int64_t k = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int K9 = 9 * kCin[l], Kp = kp_of(l);
        for (int co = 0; co < kCout[l]; ++co)
            for (int kk = 0; kk < K9; ++kk) dev[(size_t)(b.off_w[l] + (int64_t)co * Kp + kk)] = in[k++];
        for (int co = 0; co < kCout[l]; ++co) dev[(size_t)(b.off_b[l] + co)] = in[k++];
    }
    for (int c = 0; c < kFeat; ++c) dev[(size_t)(b.off_hw + c)] = in[k++];
    dev[(size_t)b.off_hb] = in[k++];
}

void free_cnn(sp_cnn *c) {
    for (Branch &b : c->br) {
        cudaFree(b.params);
        cudaFree(b.grads);
        cudaFree(b.m);
        cudaFree(b.v);
        cudaFree(b.pb);
        for (int l = 0; l < kLayers; ++l) {
            cudaFree(b.y[l]);
            cudaFree(b.dz[l]);
        }
        cudaFree(b.feat);
        cudaFree(b.logit);
        cudaFree(b.dl);
    }
    cudaFree(c->sums);
    cudaFree(c->flat);
    cudaFree(c->wpart);
    cudaFree(c->prob);
    cudaFree(c->loss);
    cudaFreeHost(c->status);
}

bool on_cnn_device(const sp_cnn *c) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return dev == c->device;
}

int upload_params(sp_cnn *c, int br, const std::vector<float> &h) {
    Branch &b = c->br[br];
    if (cudaMemcpy(b.params, h.data(), (size_t)b.n * 4, cudaMemcpyHostToDevice) != cudaSuccess) return SP_ECUDA;
    const int rc = cnn_to_bf16(b.params, b.n, b.pb, nullptr);
    if (rc) return rc;
    return cudaDeviceSynchronize() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int forward(sp_cnn *c, const __nv_bfloat16 *ft, const __nv_bfloat16 *dmt, int B, const float *labels, float *prob,
            int32_t *status, cudaStream_t st) {
    // Both branches' layers go in one launch each: with a few candidates a
    // layer is bound by its latency, not by its work.
    int rc = SP_OK;
    ConvPair p;
    p.x[0] = ft;
    p.x[1] = dmt;
    for (int l = 0; l < kLayers && !rc; ++l) {
        for (int bi = 0; bi < 2; ++bi) {
            Branch &b = c->br[bi];
            p.w[bi] = b.pb + b.off_w[l];
            p.bias[bi] = b.params + b.off_b[l];
            p.y[bi] = b.y[l];
        }
        rc = l == 0 ? cnn_conv0(p, B, kHin[l], kp_of(l), st) : cnn_conv_fwd(p, B, kHin[l], kCin[l], kp_of(l), status, st);
        p.x[0] = p.y[0];
        p.x[1] = p.y[1];
    }
    if (!rc) {
        HeadPair h;
        for (int bi = 0; bi < 2; ++bi) {
            Branch &b = c->br[bi];
            h.y[bi] = b.y[kLayers - 1];
            h.w[bi] = b.params + b.off_hw;
            h.b[bi] = b.params + b.off_hb;
            h.feat[bi] = b.feat;
            h.logit[bi] = b.logit;
        }
        rc = cnn_pool_head(h, B, ho_of(kLayers - 1) * ho_of(kLayers - 1), st);
    }
    if (!rc && labels && cudaMemsetAsync(c->loss, 0, sizeof(float), st) != cudaSuccess) rc = SP_ECUDA;
    if (!rc)
        rc = cnn_fuse_loss(c->br[0].logit, c->br[1].logit, labels, B, prob, c->br[0].dl, c->br[1].dl, c->loss, st);
    return rc;
}

int backward(sp_cnn *c, const __nv_bfloat16 *ft, const __nv_bfloat16 *dmt, int B, cudaStream_t st) {
    HeadGrad h;
    ColumnSums sums;
    for (int bi = 0; bi < 2; ++bi) {
        Branch &b = c->br[bi];
        if (cudaMemsetAsync(b.grads, 0, (size_t)b.n * 4, st) != cudaSuccess) return SP_ECUDA;
        h.feat[bi] = b.feat;
        h.dl[bi] = b.dl;
        h.w[bi] = b.params + b.off_hw;
        h.y[bi] = b.y[kLayers - 1];
        h.dz[bi] = b.dz[kLayers - 1];
        h.dw[bi] = b.grads + b.off_hw;
        h.db[bi] = b.grads + b.off_hb;
        sums.dw0[bi] = b.grads + b.off_w[0];
    }
    sums.kp0 = kp_of(0);
    int rc = cnn_head_back(h, B, ho_of(kLayers - 1) * ho_of(kLayers - 1), st);
    float *part = c->sums;
    for (int l = kLayers - 1; l >= 0 && !rc; --l) {
        const int H = kHin[l], C = kCin[l], Kp = kp_of(l);
        GradPair p{};
        for (int bi = 0; bi < 2; ++bi) {
            Branch &b = c->br[bi];
            p.x[bi] = l == 0 ? (bi == 0 ? ft : dmt) : b.y[l - 1];
            p.dz[bi] = b.dz[l];
            p.w[bi] = b.pb + b.off_w[l];
            p.dx[bi] = l == 0 ? nullptr : b.dz[l - 1];
            p.dw[bi] = b.grads + b.off_w[l];
            sums.db[bi][l] = b.grads + b.off_b[l];
        }
        sums.part[l] = part;
        sums.cols[l] = part_cols(l);
        part += (int64_t)2 * kBiasChunks * part_cols(l);
        if (l == 0) {
            rc = cnn_conv0_wgrad(p, B, H, const_cast<float *>(sums.part[l]), &sums.rows[l], st);
            break;
        }
        rc = cnn_bias_part(p, (int64_t)B * ho_of(l) * ho_of(l), kCout[l], const_cast<float *>(sums.part[l]),
                           &sums.rows[l], st);
        if (!rc) rc = cnn_conv_wgrad(p, B, H, C, Kp, c->wpart, c->status, st);
        if (!rc) rc = cnn_conv_dgrad(p, B, H, C, Kp, c->status, st);
    }
    return rc ? rc : cnn_column_sums(sums, st);
}

int check_batch(const sp_cnn *c, const void *ft, const void *dmt, int32_t B) {
    if (!c || !ft || !dmt || B < 1 || B > c->max_batch) return SP_EINVAL;
    if ((reinterpret_cast<uintptr_t>(ft) & 15) || (reinterpret_cast<uintptr_t>(dmt) & 15)) return SP_EINVAL;
    return on_cnn_device(c) ? SP_OK : SP_EINVAL;
}

// SP_ETIMEOUT, once, when a pass that the caller has waited for gave up a wait: its
// gradients are void.
int take_status(sp_cnn *c) {
    volatile int32_t *s = c->status;
    if (!*s) return SP_OK;
    *s = 0;
    c->have_grads = false;
    return SP_ETIMEOUT;
}

}  // namespace

extern "C" int64_t sp_cnn_num_params(void) { return 2 * flat_count(); }

extern "C" int sp_cnn_create(int32_t max_batch, uint64_t seed, sp_cnn **out) {
    if (!out) return SP_EINVAL;
    *out = nullptr;
    if (max_batch < 1 || max_batch > SP_CNN_MAX_BATCH) return SP_EINVAL;
    sp_cnn *c = new (std::nothrow) sp_cnn();
    if (!c) return SP_ENOMEM;
    c->max_batch = max_batch;
    int rc = cudaGetDevice(&c->device) == cudaSuccess ? SP_OK : SP_ECUDA;
    const int64_t B = max_batch;
    for (int bi = 0; bi < 2 && !rc; ++bi) {
        Branch &b = c->br[bi];
        layout(b);
        rc = dalloc((void **)&b.params, b.n * 4);
        if (!rc) rc = dalloc((void **)&b.grads, b.n * 4);
        if (!rc) rc = dalloc((void **)&b.m, b.n * 4);
        if (!rc) rc = dalloc((void **)&b.v, b.n * 4);
        if (!rc) rc = dalloc((void **)&b.pb, b.n * 2);
        for (int l = 0; l < kLayers && !rc; ++l) {
            const int64_t P = B * ho_of(l) * ho_of(l);
            rc = dalloc((void **)&b.y[l], P * kCout[l] * 2);
            if (!rc) rc = dalloc((void **)&b.dz[l], P * kCout[l] * 2);
        }
        if (!rc) rc = dalloc((void **)&b.feat, B * kFeat * 4);
        if (!rc) rc = dalloc((void **)&b.logit, B * 4);
        if (!rc) rc = dalloc((void **)&b.dl, B * 4);
        if (!rc && (cudaMemset(b.m, 0, (size_t)b.n * 4) != cudaSuccess ||
                    cudaMemset(b.v, 0, (size_t)b.n * 4) != cudaSuccess ||
                    cudaMemset(b.grads, 0, (size_t)b.n * 4) != cudaSuccess))
            rc = SP_ECUDA;
    }
    int64_t sums = 0, wpart = 0;
    for (int l = 0; l < kLayers; ++l) {
        sums += (int64_t)2 * kBiasChunks * part_cols(l);
        if (l > 0) wpart = std::max(wpart, cnn_wgrad_part_floats(max_batch, kHin[l], kCin[l], kp_of(l)));
    }
    if (!rc) rc = dalloc((void **)&c->sums, sums * 4);
    if (!rc) rc = dalloc((void **)&c->wpart, wpart * 4);
    if (!rc) rc = dalloc((void **)&c->flat, 2 * flat_count() * 4);
    if (!rc) rc = dalloc((void **)&c->prob, B * 4);
    if (!rc) rc = dalloc((void **)&c->loss, 4);
    if (!rc && cudaHostAlloc((void **)&c->status, sizeof(int32_t), cudaHostAllocPortable | cudaHostAllocMapped) !=
                   cudaSuccess) {
        cudaGetLastError();
        rc = SP_ENOMEM;
    }
    if (!rc) *c->status = 0;
    // He-normal convolution weights, zero biases, small head weights.
    std::mt19937_64 gen(seed);
    for (int bi = 0; bi < 2 && !rc; ++bi) {
        Branch &b = c->br[bi];
        std::vector<float> h((size_t)b.n, 0.f);
        for (int l = 0; l < kLayers; ++l) {
            std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / (9.0 * kCin[l])));
            for (int co = 0; co < kCout[l]; ++co)
                for (int k = 0; k < 9 * kCin[l]; ++k)
                    h[(size_t)(b.off_w[l] + (int64_t)co * kp_of(l) + k)] = (float)nd(gen);
        }
        std::normal_distribution<double> nh(0.0, 1.0 / std::sqrt((double)kFeat));
        for (int k = 0; k < kFeat; ++k) h[(size_t)(b.off_hw + k)] = (float)nh(gen);
        rc = upload_params(c, bi, h);
    }
    if (rc) {
        free_cnn(c);
        delete c;
        return rc;
    }
    *out = c;
    return SP_OK;
}

extern "C" int sp_cnn_destroy(sp_cnn *c) {
    if (!c) return SP_EINVAL;
    free_cnn(c);
    delete c;
    return SP_OK;
}

// Device values of both branches in the external order to the host: gathered by a
// kernel and copied once (a training pass with its gradients, batch 64: 861 us with
// a zeroed host copy of each branch, gathered value by value; 537 us so).
static int get_flat(const sp_cnn *c, const float *b0, const float *b1, float *h) {
    sp_cnn *m = const_cast<sp_cnn *>(c);
    std::lock_guard<std::mutex> guard(m->flat_lock);
    const int rc = cudaDeviceSynchronize() == cudaSuccess ? take_status(m) : SP_ECUDA;
    if (rc) return rc;
    FlatLayout f;
    f.segments = 0;
    auto add = [&](int64_t off, int rows, int cols, int ld) {
        f.off[f.segments] = off;
        f.rows[f.segments] = rows;
        f.cols[f.segments] = cols;
        f.ld[f.segments++] = ld;
    };
    const Branch &b = c->br[0];  // the branches are laid out alike
    for (int l = 0; l < kLayers; ++l) {
        add(b.off_w[l], kCout[l], 9 * kCin[l], kp_of(l));
        add(b.off_b[l], 1, kCout[l], kCout[l]);
    }
    add(b.off_hw, 1, kFeat, kFeat);
    add(b.off_hb, 1, 1, 1);
    const int rp = cnn_to_flat(f, b0, b1, flat_count(), m->flat, nullptr);
    if (rp) return rp;
    return cudaMemcpy(h, m->flat, (size_t)(2 * flat_count()) * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? SP_OK
                                                                                                        : SP_ECUDA;
}

extern "C" int sp_cnn_get_params(const sp_cnn *c, float *h) {
    if (!c || !h || !on_cnn_device(c)) return SP_EINVAL;
    return get_flat(c, c->br[0].params, c->br[1].params, h);
}

extern "C" int sp_cnn_set_params(sp_cnn *c, const float *h) {
    if (!c || !h || !on_cnn_device(c)) return SP_EINVAL;
    const int64_t nf = flat_count();
    for (int bi = 0; bi < 2; ++bi) {
        std::vector<float> d;
        from_flat(c->br[bi], h + bi * nf, d);
        const int rc = upload_params(c, bi, d);
        if (rc) return rc;
    }
    c->have_grads = false;
    return SP_OK;
}

extern "C" int sp_cnn_get_grads(const sp_cnn *c, float *h) {
    if (!c || !h || !c->have_grads || !on_cnn_device(c)) return SP_EINVAL;
    return get_flat(c, c->br[0].grads, c->br[1].grads, h);
}

extern "C" int sp_cnn_forward(sp_cnn *c, const void *d_ft, const void *d_dmt, int32_t batch, float *d_prob,
                              void *stream) {
    int rc = check_batch(c, d_ft, d_dmt, batch);
    if (rc) return rc;
    if (!d_prob) return SP_EINVAL;
    return forward(c, static_cast<const __nv_bfloat16 *>(d_ft), static_cast<const __nv_bfloat16 *>(d_dmt), batch,
                   nullptr, d_prob, c->status, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int sp_cnn_status(sp_cnn *c, int32_t *h_status, int32_t clear) {
    if (!c || !h_status || !on_cnn_device(c)) return SP_EINVAL;
    if (cudaDeviceSynchronize() != cudaSuccess) return SP_ECUDA;
    *h_status = *(volatile int32_t *)c->status;
    if (clear) take_status(c);
    return SP_OK;
}

extern "C" int sp_cnn_backward(sp_cnn *c, const void *d_ft, const void *d_dmt, const float *d_labels, int32_t batch,
                               float *h_loss, void *stream) {
    int rc = check_batch(c, d_ft, d_dmt, batch);
    if (rc) return rc;
    if (!d_labels) return SP_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    rc = forward(c, static_cast<const __nv_bfloat16 *>(d_ft), static_cast<const __nv_bfloat16 *>(d_dmt), batch,
                 d_labels, c->prob, c->status, st);
    if (!rc)
        rc = backward(c, static_cast<const __nv_bfloat16 *>(d_ft), static_cast<const __nv_bfloat16 *>(d_dmt), batch, st);
    if (rc) return rc;
    c->have_grads = true;
    if (!h_loss) return SP_OK;
    if (cudaMemcpyAsync(h_loss, c->loss, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SP_ECUDA;
    return take_status(c);
}

extern "C" int sp_cnn_adam_step(sp_cnn *c, float lr, void *stream) {
    if (!c || !c->have_grads || !(lr > 0.f) || !on_cnn_device(c)) return SP_EINVAL;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    ++c->step;
    for (Branch &b : c->br) {
        const int rc = cnn_adam(b.params, b.grads, b.m, b.v, b.n, lr, 0.9f, 0.999f, 1e-8f, c->step, b.pb, st);
        if (rc) return rc;
    }
    return SP_OK;
}

extern "C" int sp_cnn_train_step(sp_cnn *c, const void *d_ft, const void *d_dmt, const float *d_labels, int32_t batch,
                                 float lr, float *h_loss, void *stream) {
    int rc = sp_cnn_backward(c, d_ft, d_dmt, d_labels, batch, h_loss, stream);
    if (!rc) rc = sp_cnn_adam_step(c, lr, stream);
    return rc;
}

extern "C" int64_t sp_cnn_features_workspace_bytes(int32_t batch) {
    // a reserved block, the raw fp32 DM-time images, and 8 blocks x 4 sums per candidate
    return batch > 0 ? 2 * align256((int64_t)batch * kImg * kImg * 4) + align256((int64_t)batch * 8 * 16) : -1;
}

extern "C" int sp_cnn_features(const float *d_sub, int32_t batch, int32_t nsub, int32_t t_in, const int32_t *d_shift,
                               void *d_ft, void *d_dmt, void *d_work, int64_t work_bytes, void *stream) {
    if (!d_sub || !d_shift || !d_ft || !d_dmt || batch < 1 || nsub != kImg || t_in < kImg) return SP_EINVAL;
    if (!d_work || work_bytes < sp_cnn_features_workspace_bytes(batch) ||
        (reinterpret_cast<uintptr_t>(d_work) & 255))
        return SP_EWORKSPACE;
    float *dmt_raw = reinterpret_cast<float *>(static_cast<uint8_t *>(d_work) +
                                               align256((int64_t)batch * kImg * kImg * 4));
    float *part = reinterpret_cast<float *>(static_cast<uint8_t *>(d_work) +
                                            2 * align256((int64_t)batch * kImg * kImg * 4));
    return cnn_features(d_sub, batch, nsub, t_in, d_shift, dmt_raw, part, static_cast<__nv_bfloat16 *>(d_ft),
                        static_cast<__nv_bfloat16 *>(d_dmt), reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int sp_dmt_shifts(const double *freqs_mhz, int32_t nchan, int32_t nsub, int32_t max_sweep,
                             int32_t *h_shift) {
    if (!freqs_mhz || !h_shift || nsub < 2 || nchan < nsub || nchan % nsub || max_sweep < 0) return SP_EINVAL;
    for (int32_t c = 1; c < nchan; ++c)
        if (!(freqs_mhz[c] < freqs_mhz[c - 1]) || !(freqs_mhz[c] > 0.0)) return SP_EINVAL;
    const int32_t per = nchan / nsub;
    std::vector<double> g((size_t)nsub);
    for (int32_t s = 0; s < nsub; ++s) {
        double f = 0.0;
        for (int32_t k = 0; k < per; ++k) f += freqs_mhz[s * per + k];
        f /= per;
        g[(size_t)s] = 1.0 / (f * f);
    }
    // Eq. 1: the residual sweep of subband s is proportional to 1/f_s^2 -
    // 1/f_0^2; row j spans max_sweep * (2 j / (kImg - 1) - 1) bins across the band.
    const double span = g[(size_t)nsub - 1] - g[0];
    for (int32_t j = 0; j < kImg; ++j) {
        const double sweep = max_sweep * (2.0 * j / (kImg - 1) - 1.0);
        for (int32_t s = 0; s < nsub; ++s)
            h_shift[(int64_t)j * nsub + s] = (int32_t)std::lround(sweep * (g[(size_t)s] - g[0]) / span);
    }
    return SP_OK;
}

// Decimation of a candidate of boxcar width w: max(1, w / 4) samples per
// bin, so that the pulse spans about four bins; the window is centred on
// the boxcar's middle sample t + w / 2.
extern "C" int sp_cnn_extract(const sp_plan *plan, const uint8_t *d_staged, int64_t pitch, int64_t n_in,
                              const sp_cand *d_cands, int32_t ncand, const int32_t *h_widths, int32_t nw,
                              int32_t t_in, float *d_sub, void *stream) {
    if (!plan || !d_staged || !d_cands || ncand < 1 || ncand > 65535 || !d_sub || t_in < 1 || t_in > 4096)
        return SP_EINVAL;
    const int rc = check_widths(h_widths, nw);
    if (rc) return rc;
    if (!on_plan_device(plan) || plan->nchan % kImg || pitch < dedisp_pitch(n_in) || n_in <= 0) return SP_EINVAL;
    ExtractWidths wt;
    for (int k = 0; k < SP_MAX_WIDTHS; ++k) {
        const int32_t w = h_widths[std::min(k, nw - 1)];
        wt.dec[k] = std::max(1, w / 4);
        wt.half[k] = w / 2;
    }
    return cnn_extract(d_staged, pitch, n_in, plan->nchan, plan->d_delays, d_cands, ncand, wt, kImg, t_in, d_sub,
                       reinterpret_cast<cudaStream_t>(stream));
}

namespace sp {
int32_t cnn_max_batch(const sp_cnn *c) { return c ? c->max_batch : 0; }
int cnn_device(const sp_cnn *c) { return c ? c->device : -1; }
int cnn_forward(sp_cnn *c, const void *d_ft, const void *d_dmt, int32_t batch, float *d_prob, int32_t *status,
                cudaStream_t st) {
    const int rc = check_batch(c, d_ft, d_dmt, batch);
    if (rc) return rc;
    return forward(c, static_cast<const __nv_bfloat16 *>(d_ft), static_cast<const __nv_bfloat16 *>(d_dmt), batch,
                   nullptr, d_prob, status, st);
}
}  // namespace sp
