// cnn_tc.cu -- the classifier's convolutions on the fifth-generation tensor
// cores (arXiv 2606.27262, Sec. 3.2.2): forward, input gradients and weight
// gradients of the 3x3, stride-2 layers 1 to 4, each as an implicit GEMM with
// bf16 operands and fp32 accumulation in tensor memory.
//
// One CTA of 4 warps: warp 0 streams operands into a ring of shared-memory
// stages with tensor-memory-access copies (cp.async.bulk.tensor; a tap's operand
// is a box of the NHWC tensor, zeros outside it), warp 1 issues tcgen05.mma
// (kind::f16) and each stage's tcgen05.commit frees it for the next copy; after
// the last MMA all four warps read the accumulator from tensor memory
// (tcgen05.ld) and apply the epilogue.  blockIdx.y is the branch: both
// networks' layers run in one launch.  Every wait is bounded; a wait that runs
// out skips the epilogue, waits (bounded) for the copies and MMAs in flight and sets
// the caller's status word.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <initializer_list>
#include <mutex>

#include "sp_cnn_internal.h"

namespace sp {
namespace {

constexpr int kTcBM = 128;

// What bounds a kernel's waits, and the word it sets when one runs out (its output
// is void then).  extra: bytes the first stage expects and nothing brings (test hook).
struct Waits {
    int32_t *status;
    uint32_t extra;
    long long limit;
};
std::atomic<uint32_t> g_extra{0};
std::atomic<long long> g_limit{1LL << 31};
Waits waits(int32_t *status) { return {status, g_extra.load(), g_limit.load()}; }

__device__ __forceinline__ uint32_t s_addr32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of an operand whose rows (contiguous elements)
// are ROW bytes, in the swizzle of that width; atoms of 8 rows are 8 ROW bytes
// apart (the stride offset).  K-major operands have one row per M or N;
// MN-major ones one row per K, and blocks of ROW bytes of M or N are `lead`
// bytes apart.
template <int ROW>
__device__ __forceinline__ uint64_t row_desc(uint32_t addr, uint32_t lead = 16) {
    static_assert(ROW == 32 || ROW == 64 || ROW == 128, "swizzle width");
    constexpr uint64_t swizzle = ROW == 32 ? 6 : ROW == 64 ? 4 : 2;
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lead & 0x3FFFF) >> 4) << 16) |
           ((uint64_t)(8 * ROW / 16) << 32) | ((uint64_t)1 << 46) | (swizzle << 61);
}

// Instruction descriptor of kind::f16: D fp32, A and B bf16, M = 128, N = n;
// a_mn, b_mn: the operand is MN-major.
__host__ __device__ constexpr uint32_t mma_idesc(int n, bool a_mn = false, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcBM >> 4) << 24);
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void load_box4(const void *dst, const CUtensorMap *m, int c, int w, int h, int n, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(s_addr32(dst)),
        "l"(m), "r"(c), "r"(w), "r"(h), "r"(n), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void load_box2(const void *dst, const CUtensorMap *m, int c, int r, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            s_addr32(dst)),
        "l"(m), "r"(c), "r"(r), "r"(bar)
        : "memory");
}
// 16 accumulator columns of this warp's 32 rows.
__device__ __forceinline__ void load_acc(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 32 bytes (a sector) at a 32-byte boundary.
__device__ __forceinline__ void load32(uint32_t (&v)[8], const void *p) {
    asm volatile("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p));
}
__device__ __forceinline__ void store32(void *p, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

__device__ __forceinline__ void mbar_init_tc(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_tc(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_wait_tc(uint32_t bar, uint32_t parity, long long limit) {
    if (mbar_try_tc(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_tc(bar, parity))
        if (clock64() - t0 > limit) return false;
    return true;
}

// What the three kernels share: shared memory (stages at a multiple of 1024
// bytes, then barriers full[NS], empty[NS], done, and the tensor-memory
// address), set up by the constructor; COLS tensor-memory columns.
template <int NS, int STAGE, int COLS>
struct Pipeline {
    static constexpr int SMEM = 1024 + NS * STAGE + 8 * (2 * NS + 1) + 16;
    static_assert(STAGE % 1024 == 0 && SMEM <= 227 * 1024 && COLS >= 32 && COLS <= 512 && (COLS & (COLS - 1)) == 0,
                  "pipeline");
    uint8_t *smem;
    uint32_t *tmem_slot;
    uint32_t full0, empty0, done, tmem;
    int warp, lane;

    __device__ __forceinline__ explicit Pipeline(uint8_t *raw) {
        smem = raw + ((1024 - (s_addr32(raw) & 1023)) & 1023);
        uint64_t *bars = reinterpret_cast<uint64_t *>(smem + NS * STAGE);
        tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * NS + 1);
        full0 = s_addr32(bars);
        empty0 = s_addr32(bars + NS);
        done = s_addr32(bars + 2 * NS);
        warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr32(tmem_slot)),
                         "r"(COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (threadIdx.x == 32) {
            for (int s = 0; s < 2 * NS + 1; ++s) mbar_init_tc(full0 + 8 * s, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem = *tmem_slot;
    }
    // copy(i, stage, full barrier) issues step i's copies (and its expect);
    // multiply(i, stage address) its MMAs.  Returns whether the accumulator is
    // complete; if not, nothing is in flight any more (within the bounds of the waits).
    template <class Copy, class Multiply>
    __device__ __forceinline__ bool run(const Waits &w, int steps, Copy copy, Multiply multiply) {
        bool ok = true;
        int copied = 0;  // steps
        if (warp == 0 && lane == 0) {
            for (; copied < steps; ++copied) {
                const int s = copied % NS;
                if (copied >= NS) ok = mbar_wait_tc(empty0 + 8 * s, ((copied / NS) - 1) & 1, w.limit);
                if (!ok) break;
                copy(copied, smem + s * STAGE, full0 + 8 * s);
            }
        } else if (warp == 1 && lane == 0) {
            for (int i = 0; i < steps; ++i) {
                const int s = i % NS;
                ok = mbar_wait_tc(full0 + 8 * s, (i / NS) & 1, w.limit);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                multiply(i, s_addr32(smem + s * STAGE));
                mma_commit(empty0 + 8 * s);
            }
            mma_commit(done);  // of the MMAs that were issued
        }
        ok = mbar_wait_tc(done, 0, w.limit) && ok;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        ok = !__syncthreads_or(!ok);
        if (!ok && threadIdx.x == 0) {
            // Copies that no MMA waited for may still be landing.
            for (int i = max(0, copied - NS); i < copied; ++i) mbar_wait_tc(full0 + 8 * (i % NS), (i / NS) & 1, w.limit);
            *(volatile int32_t *)w.status = SP_STATUS_STAGING_TIMEOUT;
        }
        return ok;
    }
    __device__ __forceinline__ void finish() {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
    }
};
// First image and first row of the tile of 128 pixels from m0 (1 << lwo columns and rows an image).
__device__ __forceinline__ int tile_image(int m0, int lwo) { return m0 >> (2 * lwo); }
__device__ __forceinline__ int tile_row(int m0, int lwo) { return (m0 >> lwo) & ((1 << lwo) - 1); }

struct ConvMaps {
    CUtensorMap a[2], b[2];
};
struct ConvOut {
    const float *bias[2];
    __nv_bfloat16 *y[2];
};

// ---- forward: y = relu(conv(x) + bias) ----
// 128 output pixels x N = 2 C output channels per CTA, K = 9 taps x C input
// channels.  The 128 pixels are rows of an image (or whole images), so a tap's
// operand is one box of the input with every second column and row (the tensor
// map's element strides); the padding is the zero fill.  Bound by latency and
// L2 (the layers read 9/4 of their input).  Both branches at batch 256, layers
// 1-4: 305, 149, 104, 67 us with patches gathered by two warps (the last by
// im2col) -> 140, 61, 52, 35; at batch 5: 21, 30, 49, 38 -> 8, 9, 7, 11.
// NB: CTAs that share a tile's output channels, 2 C / NB each.
template <int C, int NB>
struct FwdShape {
    static constexpr int KC = C < 64 ? C : 64, STEPS = 9 * (C / KC), N = 2 * C / NB;  // KC channels of a tap per stage
    static constexpr int A_BYTES = kTcBM * KC * 2, B_BYTES = N * KC * 2;
    using Pipe = Pipeline<C == 16 ? 9 : C == 32 ? 6 : 4, A_BYTES + B_BYTES, N>;
};
template <int C, int NB>
__global__ void __launch_bounds__(128) conv_fwd_kernel(const __grid_constant__ ConvMaps maps, const ConvOut out, int M,
                                                       int lwo, const Waits w) {
    using S = FwdShape<C, NB>;
    extern __shared__ uint8_t smem_raw[];
    typename S::Pipe pipe(smem_raw);
    const bool branch = blockIdx.y;
    const int m0 = blockIdx.x * kTcBM, n0 = blockIdx.z * S::N;
    const bool ok = pipe.run(
        w, S::STEPS,
        [&](int i, uint8_t *stage, uint32_t full) {
            const int tap = i / (C / S::KC), c0 = (i % (C / S::KC)) * S::KC;
            expect(full, S::A_BYTES + S::B_BYTES + (i == 0 ? w.extra : 0u));
            load_box4(stage, &maps.a[branch], c0, tap % 3 - 1, 2 * tile_row(m0, lwo) + tap / 3 - 1, tile_image(m0, lwo), full);
            load_box2(stage + S::A_BYTES, &maps.b[branch], tap * C + c0, n0, full);
        },
        [&](int i, uint32_t stage) {
#pragma unroll
            for (int ks = 0; ks < S::KC / 16; ++ks)
                mma(pipe.tmem, row_desc<2 * S::KC>(stage + ks * 32), row_desc<2 * S::KC>(stage + S::A_BYTES + ks * 32),
                    mma_idesc(S::N), i > 0 || ks > 0);
        });
    if (ok) {
        // 32 columns at a time: bias, ReLU and rounding by row, then through
        // shared memory (the stages are free) so that four lanes store a row's
        // 64 bytes together.
        const int lane = pipe.lane, row0 = m0 + pipe.warp * 32;
        const float *bias = (branch ? out.bias[1] : out.bias[0]) + n0;
        __nv_bfloat16 *y = (branch ? out.y[1] : out.y[0]) + (int64_t)row0 * 2 * C + n0;
        uint4 *buf = reinterpret_cast<uint4 *>(pipe.smem) + pipe.warp * 128;
#pragma unroll 1
        for (int c0 = 0; c0 < S::N; c0 += 32) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[16], o[8];
                load_acc(pipe.tmem + ((uint32_t)(pipe.warp * 32) << 16) + (uint32_t)(c0 + 16 * half), v);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int c = c0 + 16 * half + 2 * j;
                    const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(__uint_as_float(v[2 * j]) + bias[c], 0.f),
                                                                   fmaxf(__uint_as_float(v[2 * j + 1]) + bias[c + 1], 0.f));
                    o[j] = *reinterpret_cast<const uint32_t *>(&h);
                }
                const int s = (lane >> 1) & 3;
                buf[4 * lane + ((2 * half) ^ s)] = make_uint4(o[0], o[1], o[2], o[3]);
                buf[4 * lane + ((2 * half + 1) ^ s)] = make_uint4(o[4], o[5], o[6], o[7]);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 8 * i + (lane >> 2), c = lane & 3;
                if (row0 + r < M)
                    *reinterpret_cast<uint4 *>(y + (int64_t)r * 2 * C + c0 + 8 * c) = buf[4 * r + (c ^ ((r >> 1) & 3))];
            }
            __syncwarp();
        }
    }
    pipe.finish();
}

// ---- weight gradient: part[z][branch][co][k] = sum over a range of pixels of
// dz[p][co] x[p at tap][c], k = tap * C + c ----
// M = 128 of the 9 C values of k (whole taps: 128 / C of them), N = 2 C, K =
// pixels: both operands are read as they lie, pixels being their rows, as
// MN-major operands -- no transposes and no patch matrix.  The pixels are split
// over blockIdx.z; conv_wgrad_sum_kernel adds the ranges in order, so that training
// does not depend on scheduling.  Bound by the boxes' many small rows and L2
// (9/4 of x and MT times dz).  Both branches at batch 64, layers 1-4 with the sums:
// about 1500 us with im2col, transposes and a GEMM per branch -> 112 us.
template <int C>
struct WgradShape {
    static constexpr int CO = 2 * C, TAPS = kTcBM / C, MT = (9 + TAPS - 1) / TAPS;
    static constexpr int AC = C < 64 ? C : 64, BC = CO < 64 ? CO : 64;  // channels of a box
    static constexpr int A_BOX = kTcBM * AC * 2, B_BOX = kTcBM * BC * 2;
    static constexpr int A_BYTES = kTcBM * 128 * 2, B_BYTES = kTcBM * CO * 2;
    // CTAs of both branches: one wave of as many as fit an SM (160 KB to 192 KB of stages)
    static constexpr int PER_SM = C <= 32 ? 2 : 1, CTAS = 152 * PER_SM;
    using Pipe = Pipeline<C == 64 ? 3 : 2, A_BYTES + B_BYTES, CO>;
    static int splits(int chunks) { return std::min(chunks, CTAS / (2 * MT)); }
};
template <int C>
__global__ void __launch_bounds__(128) conv_wgrad_kernel(const __grid_constant__ ConvMaps maps, int chunks,
                                                         int chunks_per_split, int lwo, int Kp, float *__restrict__ part,
                                                         const Waits w) {
    using S = WgradShape<C>;
    extern __shared__ uint8_t smem_raw[];
    typename S::Pipe pipe(smem_raw);
    const bool branch = blockIdx.y;
    const int tile = blockIdx.x, first = blockIdx.z * chunks_per_split, n = min(chunks, first + chunks_per_split) - first;
    const int ntap = min(S::TAPS, 9 - tile * S::TAPS);
    const bool ok = pipe.run(
        w, n,
        [&](int i, uint8_t *stage, uint32_t full) {
            const int m0 = (first + i) * kTcBM;
            expect(full, (uint32_t)(ntap * C / S::AC * S::A_BOX + S::B_BYTES) + (i == 0 ? w.extra : 0u));
            for (int t = 0; t < ntap; ++t) {
                const int tap = tile * S::TAPS + t;
                for (int c = 0; c < C / S::AC; ++c)
                    load_box4(stage + (t * (C / S::AC) + c) * S::A_BOX, &maps.a[branch], c * S::AC, tap % 3 - 1,
                              2 * tile_row(m0, lwo) + tap / 3 - 1, tile_image(m0, lwo), full);
            }
            for (int c = 0; c < S::CO / S::BC; ++c)
                load_box2(stage + S::A_BYTES + c * S::B_BOX, &maps.b[branch], c * S::BC, m0, full);
        },
        [&](int i, uint32_t stage) {
#pragma unroll
            for (int ks = 0; ks < kTcBM / 16; ++ks)  // 16 pixels: two atoms of 8 rows
                mma(pipe.tmem, row_desc<2 * S::AC>(stage + ks * 16 * 2 * S::AC, S::A_BOX),
                    row_desc<2 * S::BC>(stage + S::A_BYTES + ks * 16 * 2 * S::BC, S::B_BOX),
                    mma_idesc(S::CO, true, true), i > 0 || ks > 0);
        });
    if (ok) {
        const int k = tile * kTcBM + pipe.warp * 32 + pipe.lane;
        float *p = part + (int64_t)(blockIdx.z * 2 + blockIdx.y) * S::CO * Kp + k;
#pragma unroll 1
        for (int c0 = 0; c0 < S::CO; c0 += 16) {
            uint32_t v[16];
            load_acc(pipe.tmem + ((uint32_t)(pipe.warp * 32) << 16) + (uint32_t)c0, v);
            if (k < 9 * C) {
#pragma unroll
                for (int j = 0; j < 16; ++j) p[(int64_t)(c0 + j) * Kp] = __uint_as_float(v[j]);
            }
            __syncwarp();
        }
    }
    pipe.finish();
}

// ---- input gradient: dx = (transposed conv of dz) * (x > 0) ----
// 128 positions (i, j) of dz per CTA give the four input pixels (2i + ph, 2j +
// pw), each an accumulator of C columns.  Row ph = 0 takes tap row 1 of dz row i;
// ph = 1 takes tap rows 2 of row i and 0 of row i + 1; columns likewise.  So
// a step loads dz once at one of the four shifts (di, dj) and 64 of its
// channels (K), and the weights of the taps that use it (4, 2, 2 or 1), which lie
// K-row by K-row: MN-major.  No product matrix and no col2im.  Bound by memory
// (reads dz and x, writes dx) and by latency: each lane reads the mask of its four
// pixels 16 channels ahead, a 32-byte sector at a time (without: 144 us).  Both
// branches at batch 64, layers 1-4: 790 us with a GEMM and col2im per branch -> 103 us.
template <int C>
struct DgradShape {
    static constexpr int CO = 2 * C, KC = CO < 64 ? CO : 64, BC = C < 64 ? C : 64;
    static constexpr int A_BYTES = kTcBM * KC * 2, B_BOX = KC * BC * 2, B_BYTES = KC * C * 2;
    using Pipe = Pipeline<C == 16 ? 4 : 2, A_BYTES + 4 * B_BYTES, 4 * C>;
};
template <int C>
__global__ void __launch_bounds__(128) conv_dgrad_kernel(const __grid_constant__ ConvMaps maps, const ConvOut out,
                                                         const __nv_bfloat16 *__restrict__ x0,
                                                         const __nv_bfloat16 *__restrict__ x1, int M, int lwo,
                                                         const Waits w) {
    using S = DgradShape<C>;
    extern __shared__ uint8_t smem_raw[];
    typename S::Pipe pipe(smem_raw);
    const bool branch = blockIdx.y;
    const int m0 = blockIdx.x * kTcBM;
    // This lane's position and, 16 channels ahead of their use, the values of x that mask its four pixels.
    const int m = m0 + pipe.warp * 32 + pipe.lane, H = 2 << lwo;
    const int n = m >> (2 * lwo), row = (m >> lwo) & ((1 << lwo) - 1), col = m & ((1 << lwo) - 1);
    auto pixel = [&](int cls) {
        return (((int64_t)n * H + 2 * row + (cls >> 1)) * H + 2 * col + (cls & 1)) * C;
    };
    const __nv_bfloat16 *x = branch ? x1 : x0;
    uint32_t xs[4][8] = {};
    auto fetch = [&](int c0) {
        if (m < M) {
#pragma unroll
            for (int cls = 0; cls < 4; ++cls) load32(xs[cls], x + pixel(cls) + c0);
        }
    };
    fetch(0);
    // tap row (or column) u of shift d: d = 0: 1 (even pixels), 2 (odd); d = 1: 0 (odd)
    const bool ok = pipe.run(
        w, 4 * (S::CO / S::KC),
        [&](int i, uint8_t *stage, uint32_t full) {
            const int di = (i >> 1) & 1, dj = i & 1, k0 = (i >> 2) * S::KC;
            const int nu = di ? 1 : 2, nv = dj ? 1 : 2;
            expect(full, (uint32_t)(S::A_BYTES + nu * nv * S::B_BYTES) + (i == 0 ? w.extra : 0u));
            load_box4(stage, &maps.a[branch], k0, dj, tile_row(m0, lwo) + di, tile_image(m0, lwo), full);
            uint8_t *b = stage + S::A_BYTES;
            for (int u = 0; u < nu; ++u)
                for (int v = 0; v < nv; ++v) {
                    const int tap = (di ? 0 : 1 + u) * 3 + (dj ? 0 : 1 + v);
                    for (int c = 0; c < C / S::BC; ++c, b += S::B_BOX)
                        load_box2(b, &maps.b[branch], tap * C + c * S::BC, k0, full);
                }
        },
        [&](int i, uint32_t stage) {
            const int di = (i >> 1) & 1, dj = i & 1;
            const int nu = di ? 1 : 2, nv = dj ? 1 : 2;
            uint32_t b = stage + S::A_BYTES;
            for (int u = 0; u < nu; ++u)
                for (int v = 0; v < nv; ++v, b += S::B_BYTES) {
                    const int ph = di ? 1 : u, pw = dj ? 1 : v;
                    // the first use of an accumulator is at shift (0, 0), where every class has a tap
#pragma unroll
                    for (int ks = 0; ks < S::KC / 16; ++ks)
                        mma(pipe.tmem + (uint32_t)((2 * ph + pw) * C), row_desc<2 * S::KC>(stage + ks * 32),
                            row_desc<2 * S::BC>(b + ks * 16 * 2 * S::BC, S::B_BOX), mma_idesc(C, false, true),
                            i > 0 || ks > 0);
                }
        });
    if (ok) {
        __nv_bfloat16 *dx = branch ? out.y[1] : out.y[0];
#pragma unroll 1
        for (int c0 = 0; c0 < C; c0 += 16) {
            uint32_t mask[4][8];
#pragma unroll
            for (int cls = 0; cls < 4; ++cls)
#pragma unroll
                for (int q = 0; q < 8; ++q) mask[cls][q] = xs[cls][q];
            if (c0 + 16 < C) fetch(c0 + 16);
            __syncwarp();
#pragma unroll
            for (int cls = 0; cls < 4; ++cls) {
                uint32_t v[16], o[8];
                load_acc(pipe.tmem + ((uint32_t)(pipe.warp * 32) << 16) + (uint32_t)(cls * C + c0), v);
#pragma unroll
                for (int q = 0; q < 8; ++q) {  // bf16 = the upper half of an fp32
                    const float lo = __uint_as_float(mask[cls][q] << 16);
                    const float hi = __uint_as_float(mask[cls][q] & 0xFFFF0000u);
                    const __nv_bfloat162 h = __floats2bfloat162_rn(lo > 0.f ? __uint_as_float(v[2 * q]) : 0.f,
                                                                   hi > 0.f ? __uint_as_float(v[2 * q + 1]) : 0.f);
                    o[q] = *reinterpret_cast<const uint32_t *>(&h);
                }
                if (m < M) store32(dx + pixel(cls) + c0, o);
                __syncwarp();
            }
        }
    }
    pipe.finish();
}

// grads[branch][co][k] += the ranges' parts, k < 9 C: blockDim.x values a block,
// lane w of blockDim.y adding ranges w, w + blockDim.y, ... in order, then the
// lanes' sums in order.
__global__ void __launch_bounds__(256) conv_wgrad_sum_kernel(const float *__restrict__ part, int nz, int CO, int K9,
                                                             int Kp, float *__restrict__ g0, float *__restrict__ g1) {
    __shared__ float red[256];
    const int e = blockIdx.x * blockDim.x + threadIdx.x, w = threadIdx.y;  // CO * K9 is a multiple of 256
    const int co = e / K9, k = e - co * K9;
    const int64_t o = (int64_t)co * Kp + k, zs = (int64_t)2 * CO * Kp;
    const float *p = part + (int64_t)blockIdx.y * CO * Kp + o;
    float a = 0.f;
#pragma unroll 8
    for (int z = w; z < nz; z += blockDim.y) a += p[z * zs];
    red[w * blockDim.x + threadIdx.x] = a;
    __syncthreads();
    if (w) return;
    float s = 0.f;
    for (int r = 0; r < (int)blockDim.y; ++r) s += red[r * blockDim.x + threadIdx.x];
    (blockIdx.y ? g1 : g0)[o] += s;
}

// Sets a kernel's dynamic shared-memory limit once per device.
struct SmemLimit {
    std::mutex lock;
    bool configured[64] = {};
    int set(const void *kernel, int bytes) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
            cudaGetLastError();
            return SP_ECUDA;
        }
        std::lock_guard<std::mutex> guard(lock);
        if (configured[dev]) return SP_OK;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
            cudaGetLastError();
            return SP_ECUDA;
        }
        configured[dev] = true;
        return SP_OK;
    }
};

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

CUtensorMapSwizzle swizzle_of(int channels) {  // boxes of this many channels per row
    return channels == 16   ? CU_TENSOR_MAP_SWIZZLE_32B
           : channels == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                            : CU_TENSOR_MAP_SWIZZLE_128B;
}
// 128 pixels of an NHWC bf16 tensor [Nb][H][H][C]: `step` = 2 takes every second
// column and row (the box spans twice what it holds).
bool map_pixels(CUtensorMap *m, const __nv_bfloat16 *p, int Nb, int H, int C, int box_c, int step) {
    auto fn = encode_fn();
    if (!fn) return false;
    const int w = H / step, rows = std::min(w, kTcBM / w), images = kTcBM / (rows * w);
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)H, (cuuint64_t)H, (cuuint64_t)Nb};
    const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)H * C * 2, (cuuint64_t)H * H * C * 2};
    const cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)(step * w), (cuuint32_t)(step * rows), (cuuint32_t)images};
    const cuuint32_t elem[4] = {1, (cuuint32_t)step, (cuuint32_t)step, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16 *>(p), dims, strides, box, elem,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Boxes of box_c x box_r of a row-major bf16 matrix [rows][ld], `cols` columns used.
bool map_matrix(CUtensorMap *m, const __nv_bfloat16 *p, int64_t rows, int64_t cols, int64_t ld, int box_c, int box_r) {
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_c, (cuuint32_t)box_r}, elem[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(p), dims, strides, box, elem,
              CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(box_c), CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
int lwo_of(int Ho) { return Ho == 64 ? 6 : Ho == 32 ? 5 : Ho == 16 ? 4 : 3; }
int launched() {
    note_launch();
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

template <int C, int NB>
int fwd(const ConvPair &p, int Nb, int H, int Kp, const Waits &w, cudaStream_t st) {
    using S = FwdShape<C, NB>;
    ConvMaps maps;
    ConvOut out;
    for (int b = 0; b < 2; ++b) {
        if (!map_pixels(&maps.a[b], p.x[b], Nb, H, C, S::KC, 2) || !map_matrix(&maps.b[b], p.w[b], 2 * C, 9 * C, Kp, S::KC, S::N))
            return SP_ECUDA;
        out.bias[b] = p.bias[b];
        out.y[b] = p.y[b];
    }
    static SmemLimit limit;
    const int rc = limit.set(reinterpret_cast<const void *>(conv_fwd_kernel<C, NB>), S::Pipe::SMEM);
    if (rc) return rc;
    const int M = Nb * (H / 2) * (H / 2);
    conv_fwd_kernel<C, NB><<<dim3((unsigned)((M + kTcBM - 1) / kTcBM), 2, NB), 128, S::Pipe::SMEM, st>>>(maps, out, M,
                                                                                                       lwo_of(H / 2), w);
    return launched();
}

template <int C>
int wgrad(const GradPair &p, int Nb, int H, int Kp, float *part, const Waits &w, cudaStream_t st) {
    using S = WgradShape<C>;
    const int Ho = H / 2, M = Nb * Ho * Ho, chunks = (M + kTcBM - 1) / kTcBM;
    ConvMaps maps;
    for (int b = 0; b < 2; ++b)
        if (!map_pixels(&maps.a[b], p.x[b], Nb, H, C, S::AC, 2) || !map_matrix(&maps.b[b], p.dz[b], M, S::CO, S::CO, S::BC, kTcBM))
            return SP_ECUDA;
    static SmemLimit limit;
    int rc = limit.set(reinterpret_cast<const void *>(conv_wgrad_kernel<C>), S::Pipe::SMEM);
    if (rc) return rc;
    const int want = S::splits(chunks);
    const int per = (chunks + want - 1) / want, nz = (chunks + per - 1) / per;
    conv_wgrad_kernel<C><<<dim3(S::MT, 2, (unsigned)nz), 128, S::Pipe::SMEM, st>>>(maps, chunks, per, lwo_of(Ho), Kp, part,
                                                                                                w);
    rc = launched();
    if (rc) return rc;
    // Many ranges of few values (layers 1, 2) need the lanes: 18 and 14 us without; few of many are slower with them
    // (layer 4: 26 us against 10).
    const int lanes = nz >= 32 ? 8 : 1;
    conv_wgrad_sum_kernel<<<dim3(S::CO * 9 * C * lanes / 256, 2), dim3(256 / lanes, lanes), 0, st>>>(part, nz, S::CO, 9 * C, Kp, p.dw[0], p.dw[1]);
    return launched();
}

template <int C>
int dgrad(const GradPair &p, int Nb, int H, int Kp, const Waits &w, cudaStream_t st) {
    using S = DgradShape<C>;
    const int Ho = H / 2, M = Nb * Ho * Ho;
    ConvMaps maps;
    ConvOut out{};
    for (int b = 0; b < 2; ++b) {
        if (!map_pixels(&maps.a[b], p.dz[b], Nb, Ho, S::CO, S::KC, 1) || !map_matrix(&maps.b[b], p.w[b], S::CO, 9 * C, Kp, S::BC, S::KC))
            return SP_ECUDA;
        out.y[b] = p.dx[b];
    }
    static SmemLimit limit;
    const int rc = limit.set(reinterpret_cast<const void *>(conv_dgrad_kernel<C>), S::Pipe::SMEM);
    if (rc) return rc;
    conv_dgrad_kernel<C><<<dim3((unsigned)((M + kTcBM - 1) / kTcBM), 2), 128, S::Pipe::SMEM, st>>>(maps, out, p.x[0], p.x[1], M,
                                                                                                 lwo_of(Ho), w);
    return launched();
}

bool shape_ok(int Nb, int H, int C, int Kp) {
    return (C == 16 || C == 32 || C == 64 || C == 128) && (H == 128 || H == 64 || H == 32 || H == 16) && Kp >= 9 * C &&
           Kp % 8 == 0 && Nb >= 1 && (int64_t)Nb * H * H <= INT32_MAX;
}
bool aligned(std::initializer_list<const void *> ps, uintptr_t to = 16) {
    uintptr_t all = 0;
    for (const void *q : ps) all |= reinterpret_cast<uintptr_t>(q);
    return (all & (to - 1)) == 0;
}

}  // namespace

int cnn_conv_fwd(const ConvPair &p, int Nb, int H, int C, int Kp, int32_t *status, cudaStream_t st) {
    if (!shape_ok(Nb, H, C, Kp) || !aligned({p.x[0], p.x[1], p.w[0], p.w[1], p.y[0], p.y[1]})) return SP_EINVAL;
    // A few tiles leave SMs idle while each streams all of a layer's weights: where four times the CTAs still fit two
    // an SM, four share a tile's output channels (layers 3, 4 at batch 5: 11, 19 -> 7, 11 us; layer 4 at batch 64: 19 -> 13).
    const bool few = ((int64_t)Nb * (H / 2) * (H / 2) + kTcBM - 1) / kTcBM * 2 * 4 <= 2 * 152;
    const Waits w = waits(status);
    switch (C) {
        case 16: return fwd<16, 1>(p, Nb, H, Kp, w, st);
        case 32: return fwd<32, 1>(p, Nb, H, Kp, w, st);
        case 64: return few ? fwd<64, 4>(p, Nb, H, Kp, w, st) : fwd<64, 1>(p, Nb, H, Kp, w, st);
        default: return few ? fwd<128, 4>(p, Nb, H, Kp, w, st) : fwd<128, 1>(p, Nb, H, Kp, w, st);
    }
}

int64_t cnn_wgrad_part_floats(int Nb, int H, int C, int Kp) {
    const int chunks = (int)(((int64_t)Nb * (H / 2) * (H / 2) + kTcBM - 1) / kTcBM);
    const int nz = C == 16   ? WgradShape<16>::splits(chunks)
                   : C == 32 ? WgradShape<32>::splits(chunks)
                   : C == 64 ? WgradShape<64>::splits(chunks)
                             : WgradShape<128>::splits(chunks);
    return (int64_t)nz * 2 * 2 * C * Kp;
}

int cnn_conv_wgrad(const GradPair &p, int Nb, int H, int C, int Kp, float *part, int32_t *status, cudaStream_t st) {
    if (!shape_ok(Nb, H, C, Kp) || !aligned({p.x[0], p.x[1], p.dz[0], p.dz[1]})) return SP_EINVAL;
    const Waits w = waits(status);
    switch (C) {
        case 16: return wgrad<16>(p, Nb, H, Kp, part, w, st);
        case 32: return wgrad<32>(p, Nb, H, Kp, part, w, st);
        case 64: return wgrad<64>(p, Nb, H, Kp, part, w, st);
        default: return wgrad<128>(p, Nb, H, Kp, part, w, st);
    }
}

int cnn_conv_dgrad(const GradPair &p, int Nb, int H, int C, int Kp, int32_t *status, cudaStream_t st) {
    if (!shape_ok(Nb, H, C, Kp) || !aligned({p.dz[0], p.dz[1], p.w[0], p.w[1]}) ||
        !aligned({p.x[0], p.x[1], p.dx[0], p.dx[1]}, 32))
        return SP_EINVAL;
    const Waits w = waits(status);
    switch (C) {
        case 16: return dgrad<16>(p, Nb, H, Kp, w, st);
        case 32: return dgrad<32>(p, Nb, H, Kp, w, st);
        case 64: return dgrad<64>(p, Nb, H, Kp, w, st);
        default: return dgrad<128>(p, Nb, H, Kp, w, st);
    }
}

void set_tc_fault(uint32_t extra_bytes, long long wait_limit) {
    g_extra = extra_bytes;
    g_limit = wait_limit;
}

}  // namespace sp
