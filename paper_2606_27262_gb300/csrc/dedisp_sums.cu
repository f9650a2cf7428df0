// dedisp_sums.cu -- shared-sum dedispersion on sm_103a (arXiv 2606.27262,
// Sec. 3.1.1): the DM transform out[d][t] = sum_c in[t + delay[d][c]][c] with
// the sums that several trial DMs share formed once.
//
// The DMs of a tile see a group of up to 16 neighbouring channels at few
// distinct relative delays (plan_sums.cpp), so per group
//   row_p[j] = sum_i in[t0 + base + j + r_p[i]][c0 + i]       per pattern p,
//   out[d][t0 + t] += row_{p(d)}[delay[d][c0] - base + t]     per DM d,
// exact in integers.  A direct sum reads one staged byte per channel, DM and
// sample; here a DM reads two bytes per GROUP and sample, and the rows cost
// about a channel's loads each.
//
// What bounds it: the SM's shared-memory data pipe (78 % busy over the
// 5751-trial, 4096-channel plan: 43 % of its wavefronts are the DMs'
// reads of the rows, the rest makes the rows) and instruction issue (67 %).
// That plan over 131072 samples: 133 ms with the direct kernel, 45.5 ms here;
// 64 x 1024 because a tile's 65536 packed sums take half the registers, and
// rows serve more DMs, and waste less on the spread of their delays, the larger
// the tile is (modelled: 128 x 512 18 % slower, 32 x 2048 12 %, two CTAs of
// 64 x 512 9 %).  Measured and not taken: 16 consumer and 4 producer warps (80
// ms; too few independent producers), 8 producers (56), rows over a group's
// whole spread instead of what their DMs read (53), four smaller slots (52).
//
// One CTA (one per SM) = up to 64 DMs x 1024 samples, 20 warps:
//   8 consumer warps   8 DMs x 1024 samples each as packed 16-bit sums (word j
//                      holds samples j and j + 512, so that a row at any
//                      sample offset is read by aligned, conflict-free 32-bit
//                      loads): one shared load and one add per two samples of
//                      a group.  After at most 256 channels the high bytes of
//                      the sums move to carries in tensor memory (128 words
//                      per thread), so that nothing returns to global memory
//                      before the tile is done.
//   11 producer warps  form the rows, a job being one segment of a group's path
//                      for 128 samples and the 128 samples 512 later: four
//                      consecutive samples per lane and half in registers as
//                      S = sum of the 4-byte words and H = sum of their odd
//                      bytes, one channel moved by one sample per step, one
//                      16-byte store per row.
//   1 loader warp      bulk copies (TMA) of the channels' windows and the
//                      producers' program, up to three chunks ahead.
// Row slots and raw slots are rings of three, handed over by mbarriers:
// raw_full[s] (bytes landed), full[s] (all jobs of the chunk done; also frees
// the raw slot), empty[s] (all consumers done).  Every wait is bounded; a wait
// that runs out raises `failed`, every role leaves its loop, the loader waits
// (bounded) for its copies in flight and the status bit is set.
#include <mutex>

#include "sp_internal.h"

namespace sp {
namespace {

constexpr int kConsumers = 8, kProducers = 11;
constexpr int kThreads = 32 * (kConsumers + kProducers + 1);  // and the loader
constexpr int kGroupTiles = kDedispTileGroupDms / kSumDms;  // DM tiles per raster group
// Registers: 96 a thread at launch (640 threads); the consumer warpgroups
// take 160 (128 of them sums), the other three keep 48:
// 256 * 160 + 384 * 48 <= 640 * 96.
constexpr int kLaunchRegs = 96, kConsumerRegs = 160, kProducerRegs = 48;
static_assert(32 * kConsumers * kConsumerRegs + 32 * (kProducers + 1) * kProducerRegs <= kThreads * kLaunchRegs &&
                  kConsumers % 4 == 0 && (kProducers + 1) % 4 == 0,
              "register split");
// A producer takes every kProducers-th job, so it has one in at least every
// third chunk, as its waits need (see produce).
static_assert(kProducers <= 3 * kSumMinJobs, "producer gap");
constexpr int kTmemCols = 256;  // 2 consumer warps per lane quarter x 128 words
static_assert(kSumDms == 8 * kConsumers && kSumTime == 1024, "consumer layout");
// header: raw_full[3], full[3], empty[3], failed, tensor-memory address
constexpr int kFailedOffset = 96, kTmemOffset = 100;
static_assert(8 * 3 * kSumSlots <= kFailedOffset, "header");

__device__ long long g_sums_wait_limit = 1LL << 31;  // test hook, see set_sums_fault
__device__ uint32_t g_sums_extra_bytes = 0;

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return done != 0;
}
__device__ __forceinline__ void arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Bounded wait; gives up when another role has failed, too.
__device__ __forceinline__ bool slow_wait(uint32_t bar, uint32_t parity, volatile int *failed) {
    const long long t0 = clock64();
    const long long limit = *(volatile long long *)&g_sums_wait_limit;
    while (!try_wait(bar, parity)) {
        if (*failed) return false;
        if (clock64() - t0 > limit) {
            *failed = 1;
            return false;
        }
    }
    return true;
}
// Warp-uniform: every lane waits, and all lanes agree on the outcome.
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, volatile int *failed) {
    bool ok = try_wait(bar, parity);
    if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, ok || slow_wait(bar, parity, failed));
    else ok = true;
    return ok;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ uint32_t odd_bytes(uint32_t w) { return __byte_perm(w, 0u, 0x4341); }

// 8 words of a thread's carries in tensor memory.
__device__ __forceinline__ void tmem_load8(uint32_t a, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(a));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_store8(uint32_t a, const uint32_t (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(a)
                 : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// The CTA's work item, in the header of shared memory.
struct Item {
    const SumTablesDev *tab;
    const uint8_t *xt;
    int64_t pitch, n_out, t0;
    int32_t *out;
    int32_t tile, d_first, d_cnt;
};
constexpr int kItemOffset = 128;
static_assert(kItemOffset + (int)sizeof(Item) <= kSumHeader && kTmemOffset + 4 <= kItemOffset, "header");
__device__ __forceinline__ const volatile Item &item_of(const uint8_t *smem) {
    return *reinterpret_cast<const volatile Item *>(smem + kItemOffset);
}

// ---- loader: one warp ----
__device__ __forceinline__ void load_chunks(uint8_t *smem, volatile int *failed) {
    const int lane = threadIdx.x & 31;
    const SumTablesDev *tab = item_of(smem).tab;
    const uint8_t *xt = item_of(smem).xt;
    const int64_t pitch = item_of(smem).pitch, t0 = item_of(smem).t0;
    const int tile = item_of(smem).tile;
    const int first = __ldg(tab->tile_chunk + tile), n = __ldg(tab->tile_chunk + tile + 1) - first;
    const uint32_t bars = saddr(smem), raw0 = bars + kSumHeader;
    // A chunk's geometry is fetched while the chunk before it is awaited, and
    // its descriptor a chunk earlier still: neither latency delays a copy.
    auto chunk = [&](int i) { return __ldg(tab->chunks + first + min(i, n - 1)); };
    auto prog_bytes = [&](int i) { return (uint32_t)__ldg(tab->prog_bytes + first + min(i, n - 1)); };
    auto geo_of = [&](const int4 &c) {
        return lane < c.x ? __ldg(tab->geo + c.z + lane) : make_int4(0, 0, 0, 0);
    };
    int4 ch = chunk(0), ch1 = chunk(1), g = geo_of(ch);
    uint32_t pbytes = prog_bytes(0), pbytes1 = prog_bytes(1);
    int k = 0;
    for (; k < n; ++k) {
        const int s = k % kSumSlots;
        const uint32_t bar = bars + 8 * s, slot = raw0 + s * kSumRawBytes;
        if (k >= kSumSlots && !wait(bars + 8 * (kSumSlots + s), (k / kSumSlots - 1) & 1, failed)) break;
        // Bytes of this channel's window inside the staged row (past it only
        // samples that no output needs).
        const int64_t at = t0 + g.x;
        const uint32_t bytes = lane < ch.x ? (uint32_t)min((int64_t)g.y, pitch - at) : 0u;
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes) + pbytes;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"(total + (k == 0 ? g_sums_extra_bytes : 0u))
                         : "memory");
        __syncwarp();
        if (lane < ch.x) bulk_load(slot + g.z, xt + (int64_t)(ch.y + lane) * pitch + at, bytes, bar);
        if (lane == 31) bulk_load(slot, tab->prog + ch.w, pbytes, bar);
        ch = ch1;
        pbytes = pbytes1;
        g = geo_of(ch);
        ch1 = chunk(k + 2);
        pbytes1 = prog_bytes(k + 2);
    }
    // No copy may land after the CTA has left: bounded waits for the last
    // chunk issued into each slot (already complete unless a wait ran out).
    for (int j = max(0, k - kSumSlots); j < k; ++j) {
        const long long w0 = clock64();
        const long long limit = *(volatile long long *)&g_sums_wait_limit;
        while (!try_wait(bars + 8 * (j % kSumSlots), (j / kSumSlots) & 1))
            if (clock64() - w0 > limit) break;
    }
}

// ---- producers: eleven warps ----
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {  // low 16 bits of sel
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
// One job: a segment's rows for the 32 quads from quad q0; the lane's samples
// are 4q .. 4q + 3 of the rows and the four kSumHalf later.
//   prog  the segment: {channels | steps << 16, row, lanes, last quad}, {raw
//         offset, selector} per channel (an even number), {raw offset, old
//         selector | row << 16, new selector, lanes} per step, and four idle
//         steps; row = where the pass's first quad lies in the row slot, in
//         units of 16 bytes, lanes = which quads to store (0: not complete).
__device__ __forceinline__ void make_rows(const uint8_t *raw, uint8_t *rows, const uint4 *prog, int q0) {
    const uint4 head = *prog++;
    const int ninit = (int)(head.x & 0xFFFFu), nsteps = (int)(head.x >> 16), lane = threadIdx.x & 31;
    const uint8_t *src = raw + 4 * min(q0 + lane, (int)head.w);
    const uint32_t me = 1u << lane;
    rows += 16 * lane;
    uint32_t S0 = 0, S1 = 0, H0 = 0, H1 = 0;
    auto word = [&](uint32_t off) { return *reinterpret_cast<const uint32_t *>(src + off); };
    // The first row: two channels per entry.
    for (int i = 0; i < ninit; i += 2, ++prog) {
        const uint4 o = *prog;
        const uint32_t xa = prmt(word(o.x), word(o.x + 4), o.y);
        const uint32_t ya = prmt(word(o.x + kSumHalf), word(o.x + kSumHalf + 4), o.y);
        uint32_t xb = prmt(word(o.z), word(o.z + 4), o.w);
        uint32_t yb = prmt(word(o.z + kSumHalf), word(o.z + kSumHalf + 4), o.w);
        if (i + 1 >= ninit) xb = yb = 0u;
        S0 += xa + xb;
        S1 += ya + yb;
        H0 += odd_bytes(xa) + odd_bytes(xb);
        H1 += odd_bytes(ya) + odd_bytes(yb);
    }
    auto store = [&](int32_t row, uint32_t lanes) {
        // 16-bit lanes (j, j + 2) of both halves -> words (j, j + kSumHalf)
        const uint32_t E0 = S0 - (H0 << 8), E1 = S1 - (H1 << 8);
        const uint4 v = make_uint4(prmt(E0, E1, 0x5410), prmt(H0, H1, 0x5410), prmt(E0, E1, 0x7632),
                                   prmt(H0, H1, 0x7632));
        if (lanes & me) *reinterpret_cast<uint4 *>(rows + 16 * row) = v;
    };
    store((int32_t)head.y, head.z);
    // Steps, two entries in registers and the next step's words in flight.
    uint4 e0 = prog[0], e1 = prog[1];
    prog += 2;
    uint32_t w0, w1, v0, v1;
    auto fetch = [&](uint32_t off) {
        w0 = word(off);
        w1 = word(off + 4);
        v0 = word(off + kSumHalf);
        v1 = word(off + kSumHalf + 4);
    };
    fetch(e0.x);
    auto step = [&](uint4 &e, const uint4 &next) {
        const uint32_t o0 = prmt(w0, w1, e.y), n0 = prmt(w0, w1, e.z);
        const uint32_t o1 = prmt(v0, v1, e.y), n1 = prmt(v0, v1, e.z);
        fetch(next.x);
        const int32_t row = (int32_t)e.y >> 16;
        const uint32_t lanes = e.w;
        e = *prog++;
        S0 += n0 - o0;
        S1 += n1 - o1;
        H0 += odd_bytes(n0) - odd_bytes(o0);
        H1 += odd_bytes(n1) - odd_bytes(o1);
        store(row, lanes);
    };
#pragma unroll 1
    for (int s = 0; s < nsteps; s += 2) {
        step(e0, e1);
        if (s + 1 >= nsteps) break;
        step(e1, e0);
    }
}

// Producer pw takes jobs pw, pw + kProducers, ... of the tile.  A job waits for its row
// slot before its raw slot: a producer may skip up to two chunks, and only
// empty[] of the chunk three back proves that the raw slot's earlier phase is
// over (a parity wait two phases early would pass).
__device__ __forceinline__ void produce(uint8_t *smem, int pw, volatile int *failed) {
    const uint32_t bars = saddr(smem);
    uint8_t *raw0 = smem + kSumHeader, *row0 = raw0 + kSumSlots * kSumRawBytes;
    const uint2 *job;
    int n;
    {
        const SumTablesDev *tab = item_of(smem).tab;
        const int tile = item_of(smem).tile, j0 = __ldg(tab->tile_job + tile);
        n = __ldg(tab->tile_job + tile + 1) - j0;
        job = tab->jobs + j0;
    }
    uint2 next = pw < n ? __ldg(job + pw) : make_uint2(0u, 0u);
    for (int j = pw; j < n; j += kProducers) {
        const uint2 d = next;
        if (j + kProducers < n) next = __ldg(job + j + kProducers);
        const uint32_t s = d.x & 3u, parity = (d.x >> 2) & 1u;
        if (!(d.x & kSumJobFirstUse) && !wait(bars + 8 * (2 * kSumSlots + s), parity ^ 1u, failed)) return;
        if (!wait(bars + 8 * s, parity, failed)) return;
        const uint8_t *raw = raw0 + s * kSumRawBytes;
        make_rows(raw, row0 + s * kSumRowBytes, reinterpret_cast<const uint4 *>(raw) + (d.y & 0xFFFFu), (int)(d.y >> 16));
        __syncwarp();
        if ((threadIdx.x & 31) == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bars + 8 * (kSumSlots + s)),
                         "r"(d.x >> 8)
                         : "memory");
    }
}

// ---- consumers: eight warps ----
__device__ __forceinline__ void consume(uint8_t *smem, uint32_t tmem, volatile int *failed) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool active = 8 * warp < item_of(smem).d_cnt;
    const uint32_t bars = saddr(smem);
    const uint32_t row0 = bars + kSumHeader + kSumSlots * kSumRawBytes + 4 * lane;
    int left;  // groups
    const int4 *off;
    {
        const SumTablesDev *tab = item_of(smem).tab;
        const int tile = item_of(smem).tile, g0 = __ldg(tab->tile_group + tile);
        left = __ldg(tab->tile_group + tile + 1) - g0;
        off = reinterpret_cast<const int4 *>(tab->off + (int64_t)g0 * kSumDms + 8 * warp);
    }
    const uint32_t my_tmem = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 128u * (uint32_t)(warp >> 2);
    uint32_t A[8][16];  // word 32 q + lane of DM i
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 16; ++q) A[i][q] = 0u;
    bool carried = false, fresh = true;  // fresh: the next group starts a chunk
    int s = 0;                           // slot
    uint32_t parity = 0;
    int4 o0 = __ldg(off), o1 = __ldg(off + 1);
    for (; left > 0; --left) {
        const int flags = o0.x & 3;
        if (fresh && !wait(bars + 8 * (kSumSlots + s), parity, failed)) return;
        fresh = false;
        off += left > 1 ? kSumDms / 4 : 0;
        // Loads run two batches of four words ahead of the adds, so that both go on at once.
        const uint32_t rows = row0 + s * kSumRowBytes;
        uint32_t w[3][4];
        auto load = [&](const int4 &o, int b) {  // batch b: words 4 (b % 4) .. of the half's DM b / 4
            const uint32_t r = rows + (uint32_t)(b / 4 == 0 ? o.x : b / 4 == 1 ? o.y : b / 4 == 2 ? o.z : o.w);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[b % 3][j]) : "r"(r + 128u * (4 * (b & 3) + j)));
        };
        auto add4 = [&](const int4 &o, int i0) {
            load(o, 0);
            load(o, 1);
#pragma unroll
            for (int b = 0; b < 16; ++b) {
                if (b + 2 < 16) load(o, b + 2);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    A[i0 + b / 4][4 * (b & 3) + j] += w[b % 3][j];
            }
        };
        // Each half of the offsets is replaced by the next group's as soon as it has been used.
        if (active) {
            o0.x -= flags;
            add4(o0, 0);
            o0 = __ldg(off);
            add4(o1, 4);
            o1 = __ldg(off + 1);
        } else {
            o0 = __ldg(off);
        }
        if (flags & kSumLastOfChunk) {
            __syncwarp();
            if (lane == 0) arrive(bars + 8 * (2 * kSumSlots + s));
            if (++s == kSumSlots) {
                s = 0;
                parity ^= 1u;
            }
            fresh = true;
        }
        if (flags & kSumCarryAfter) {
            // The lanes' high bytes go to the carries; at most 255 stays.
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                uint32_t c[8];
                if (carried) {
                    tmem_load8(my_tmem + 8 * k, c);
                } else {
#pragma unroll
                    for (int q = 0; q < 8; ++q) c[q] = 0u;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    uint32_t &v = A[k >> 1][8 * (k & 1) + q];
                    c[q] += odd_bytes(v);
                    v &= 0x00FF00FFu;
                }
                tmem_store8(my_tmem + 8 * k, c);
            }
            carried = true;
        }
    }
    const int d_cnt = item_of(smem).d_cnt - 8 * warp, d0 = item_of(smem).d_first + 8 * warp;
    const int64_t n_out = item_of(smem).n_out, t = item_of(smem).t0 + lane;
    int32_t *const out = item_of(smem).out + t;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int i = k >> 1;
        if (i >= d_cnt) break;
        uint32_t c[8];
        if (carried) {
            tmem_load8(my_tmem + 8 * k, c);
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) c[q] = 0u;
        }
        int32_t *o = out + (int64_t)(d0 + i) * n_out;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = 32 * (8 * (k & 1) + q);
            const uint32_t v = A[i][8 * (k & 1) + q];
            if (t + j < n_out) o[j] = (int32_t)((v & 0xFFFFu) + ((c[q] & 0xFFFFu) << 8));
            if (t + j + kSumHalf < n_out) o[j + kSumHalf] = (int32_t)((v >> 16) + ((c[q] >> 16) << 8));
        }
    }
}

__device__ __forceinline__ void sums_tile(uint8_t *smem, const SumTablesDev *tab, const uint8_t *xt, int64_t pitch,
                                          int64_t n_out, int32_t *out, int tile, int64_t t0,
                                          int32_t *__restrict__ status) {
    const int warp = threadIdx.x >> 5;
    volatile int *failed = reinterpret_cast<volatile int *>(smem + kFailedOffset);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kTmemOffset);
    const bool carries = tab->nchan > kSumCarryChannels;
    if (threadIdx.x < 3 * kSumSlots) {
        const int kind = threadIdx.x / kSumSlots;
        const uint32_t count = kind == 0 ? 1u : kind == 1 ? (uint32_t)kSumJobArrivals : (uint32_t)kConsumers;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(smem) + 8 * threadIdx.x), "r"(count) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        *failed = 0;
        Item *it = reinterpret_cast<Item *>(smem + kItemOffset);
        *it = Item{tab, xt, pitch, n_out, t0, out, tile, __ldg(tab->tile_first + tile), __ldg(tab->tile_count + tile)};
    }
    if (carries && warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp < kConsumers) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsumerRegs));
        consume(smem, carries ? *tmem_slot : 0u, failed);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProducerRegs));
        if (warp < kConsumers + kProducers) produce(smem, warp - kConsumers, failed);
        else load_chunks(smem, failed);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0 && item_of(smem).tab->nchan > kSumCarryChannels)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(kTmemCols) : "memory");
    if (threadIdx.x == 0 && *failed) atomicOr(status, SP_STATUS_STAGING_TIMEOUT);
}

// Groups of DM tiles sweep all time tiles together, so that the CTAs resident
// at one time read overlapping windows from L2.
__device__ __forceinline__ void raster(int64_t id, int ntiles, int64_t ntime, int &tile, int64_t &tq) {
    const int64_t per_group = (int64_t)kGroupTiles * ntime;
    const int group = (int)(id / per_group);
    const int64_t r = id - group * per_group;
    const int width = min(kGroupTiles, ntiles - group * kGroupTiles);
    tile = group * kGroupTiles + (int)(r % width);
    tq = r / width;
}

__global__ void __launch_bounds__(kThreads, 1)
dedisp_sums_kernel(const uint8_t *__restrict__ xt, int64_t pitch, int64_t n_out, int32_t *__restrict__ out,
                   const SumTablesDev *__restrict__ tables, int64_t ntime, int32_t *__restrict__ status) {
    extern __shared__ __align__(128) uint8_t smem[];
    int tile;
    int64_t tq;
    raster((int64_t)blockIdx.x, tables->ntiles, ntime, tile, tq);
    sums_tile(smem, tables, xt, pitch, n_out, out, tile, tq * kSumTime, status);
}

// The same tile for work item blockIdx.x of several beams (items numbered
// beam by beam, each beam in raster order).
__global__ void __launch_bounds__(kThreads, 1)
dedisp_sums_items_kernel(const BatchBeamDev *__restrict__ beams, const int64_t *__restrict__ item_begin,
                         int32_t nbeams, int32_t *__restrict__ status) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int64_t item = blockIdx.x;
    int lo = 0, hi = nbeams - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(item_begin + mid) <= item) lo = mid;
        else hi = mid - 1;
    }
    const BatchBeamDev bm = beams[lo];
    int tile;
    int64_t tq;
    raster(item - __ldg(item_begin + lo), bm.sums->ntiles, (int64_t)bm.ntime, tile, tq);
    sums_tile(smem, bm.sums, bm.xt, bm.pitch, bm.n_out, bm.out, tile, tq * kSumTime, status);
}

constexpr int kMaxDev = 64;
std::mutex g_lock;
bool g_configured[kMaxDev] = {};

}  // namespace

int sums_configure() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SP_ECUDA;
    if (dev < 0 || dev >= kMaxDev) return SP_ELIMIT;
    std::lock_guard<std::mutex> guard(g_lock);
    if (g_configured[dev]) return SP_OK;
    if (cudaFuncSetAttribute(dedisp_sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumSmem) != cudaSuccess ||
        cudaFuncSetAttribute(dedisp_sums_items_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumSmem) !=
            cudaSuccess) {
        cudaGetLastError();
        return SP_ECUDA;
    }
    g_configured[dev] = true;
    return SP_OK;
}

int set_sums_fault(uint32_t extra_bytes, long long wait_limit) {
    if (cudaMemcpyToSymbol(g_sums_extra_bytes, &extra_bytes, sizeof extra_bytes) != cudaSuccess ||
        cudaMemcpyToSymbol(g_sums_wait_limit, &wait_limit, sizeof wait_limit) != cudaSuccess) {
        cudaGetLastError();
        return SP_ECUDA;
    }
    return SP_OK;
}

int launch_dedisperse_sums(const sp_plan *plan, const uint8_t *d_xt, int64_t pitch, int64_t n_out, int32_t *d_out,
                           cudaStream_t stream, int32_t *status) {
    int rc = sums_configure();
    if (rc) return rc;
    const int64_t ntime = (n_out + kSumTime - 1) / kSumTime;
    dedisp_sums_kernel<<<(unsigned)(ntime * plan->sums_ntiles), kThreads, kSumSmem, stream>>>(
        d_xt, pitch, n_out, d_out, plan->d_sums, ntime, status ? status : plan->d_status);
    note_launch(1, 1);
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

int launch_dedisperse_sums_batch(const BatchLaunch &b, cudaStream_t stream) {
    if (b.nitems < 1 || b.nitems > INT32_MAX) return b.nitems < 1 ? SP_EINVAL : SP_ELIMIT;
    int rc = sums_configure();
    if (rc) return rc;
    dedisp_sums_items_kernel<<<(unsigned)b.nitems, kThreads, kSumSmem, stream>>>(b.d_beams, b.d_item_begin, b.nbeams,
                                                                               b.d_status);
    note_launch(1, 1);
    return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ECUDA;
}

}  // namespace sp
