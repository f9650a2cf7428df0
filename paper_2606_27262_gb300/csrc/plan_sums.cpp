// plan_sums.cpp -- tables of the shared-sum dedispersion kernel
// (dedisp_sums.cu; arXiv 2606.27262, Sec. 3.1.1: the DM transform).
//
// The trial DMs of a tile see a group of neighbouring channels at few
// distinct relative delays: channel i of the group arrives r = delay[d][i] -
// delay[d][0] samples after the first, and over 64 consecutive trials the
// vector r takes far fewer than 64 values (on the 5751-trial, 4096-channel
// plan at DM steps of 0.1: 4 for groups of 4 channels, 8 for 8, 19 for 16).
// The group's sum over one such pattern is a time series that every DM of
// the pattern adds at its own offset.  The sums are integers, so the result is
// that of the direct sum, bit for bit.
//
// A pattern's row is made from the previous one by moving single channels by
// one sample (most neighbouring patterns differ in one channel), so a row
// costs about one channel's loads instead of the whole group's.  A row covers
// only the samples that some DM of its pattern reads; each 128-sample pass
// over a group has its own path through the patterns that need it.  Here the
// patterns of each group are found, their paths laid out, the group size is
// chosen per 16 channels by modelled clocks, and groups are packed into chunks.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>

#include "sp_internal.h"

namespace sp {
namespace {

constexpr int kMaxDms = kSumDms;

// One group of channels in one tile.
struct Group {
    int32_t c0 = 0, n = 0;            // channels
    int32_t base = 0, spread = 0;     // smallest delay of channel c0 over the tile, and its range
    int32_t quads = 0;                // quads (4 words) that the rows reach over
    int32_t npat = 0;
    int64_t row_quads = 0;            // sum of the rows' own quads
    int32_t inits = 0, steps = 0, rows = 0, jobs = 0;  // summed over the passes
    int8_t pat_of[kMaxDms];           // pattern of each DM
    int32_t r[kMaxDms][kSumMaxGroup]; // relative delays of the patterns
    int32_t qs[kMaxDms], qe[kMaxDms]; // quads of each pattern's row
    // Paths: per pass a run of (pattern, starts a segment) entries.
    struct Visit {
        int8_t pat;
        bool fresh;
    };
    std::vector<Visit> path;
    std::vector<int32_t> pass_end;    // [passes] end of each pass's entries
    int passes() const { return (quads + 31) / 32; }
    int64_t row_bytes() const { return row_quads * 16; }
    // Whether a row slot takes the rows and a raw slot a window of this reach.
    bool may_fit() const { return row_bytes() <= kSumRowBytes && quads <= kSumRawBytes / 4; }
};

// Modelled SM clocks of a group: shared-memory wavefronts (128 bytes a clock;
// per pass two words and two halves per initial channel or step, the entries
// that describe them, a 16-byte store per row; per DM and word one), plus an
// eighth of the warp instructions (four a clock, half hidden).
double group_clocks(const Group &g, int cnt) {
    const double warps = (cnt + 7) / 8;
    const double wf = 4.5 * g.inits + 5.0 * g.steps + 4.0 * g.rows + 2.0 * g.jobs + 136.0 * warps;
    const double ins = 16.0 * g.inits + 35.0 * g.steps + 60.0 * g.jobs + 290.0 * warps;
    return wf + ins / 8.0;
}
constexpr double kChunkClocks = 100.0;

void analyse(const sp_plan &p, int32_t d0, int cnt, int32_t c0, int n, Group &g) {
    g.c0 = c0;
    g.n = n;
    int32_t lo = INT32_MAX, hi = 0, bmin[kMaxDms], bmax[kMaxDms];
    g.npat = 0;
    for (int d = 0; d < cnt; ++d) {
        const int32_t *row = &p.delays[(size_t)(d0 + d) * p.nchan + c0];
        lo = std::min(lo, row[0]);
        hi = std::max(hi, row[0]);
        int32_t v[kSumMaxGroup];
        for (int i = 0; i < n; ++i) v[i] = row[i] - row[0];
        int k = 0;
        while (k < g.npat && std::memcmp(g.r[k], v, sizeof(int32_t) * n)) ++k;
        if (k == g.npat) {
            std::memcpy(g.r[g.npat++], v, sizeof(int32_t) * n);
            bmin[k] = bmax[k] = row[0];
        }
        bmin[k] = std::min(bmin[k], row[0]);
        bmax[k] = std::max(bmax[k], row[0]);
        g.pat_of[d] = (int8_t)k;
    }
    g.base = lo;
    g.spread = hi - lo;
    g.quads = (kSumHalf + g.spread + 3) / 4;
    g.row_quads = 0;
    for (int k = 0; k < g.npat; ++k) {
        g.qs[k] = (bmin[k] - lo) / 4;
        g.qe[k] = (bmax[k] - lo + kSumHalf + 3) / 4;
        g.row_quads += g.qe[k] - g.qs[k];
    }
    if (!g.may_fit()) return;  // no paths for a group that no slot takes: it may have millions of passes
    // Moves from one pattern to another: channels that differ, if each does by
    // one sample.
    constexpr int kFar = 255;
    uint8_t moves[kMaxDms][kMaxDms];
    for (int a = 0; a < g.npat; ++a) {
        moves[a][a] = 0;
        for (int b = a + 1; b < g.npat; ++b) {
            int h = 0;
            for (int i = 0; i < n; ++i) {
                const int diff = g.r[b][i] - g.r[a][i];
                h += diff == 0 ? 0 : (diff == 1 || diff == -1) ? 1 : kFar;
            }
            moves[a][b] = moves[b][a] = (uint8_t)std::min(h, kFar);
        }
    }
    // Per pass: from each row to the nearest pattern left (fewest moves); a
    // new segment, summed from all its channels, where none is within n.
    g.path.clear();
    g.pass_end.clear();
    g.inits = g.steps = g.rows = g.jobs = 0;
    for (int pass = 0; pass < g.passes(); ++pass) {
        int todo[kMaxDms], left = 0;
        for (int k = 0; k < g.npat; ++k)
            if (g.qs[k] < 32 * pass + 32 && g.qe[k] > 32 * pass) todo[left++] = k;
        g.rows += left;
        int cur = -1;
        while (left > 0) {
            int best = 0, bd = kFar + 1;
            for (int j = 0; j < left && cur >= 0; ++j)
                if (moves[cur][todo[j]] < bd) {
                    bd = moves[cur][todo[j]];
                    best = j;
                }
            const bool fresh = cur < 0 || bd > n;
            if (fresh) {
                best = 0;
                g.inits += n;
                ++g.jobs;
            } else {
                g.steps += bd;
            }
            cur = todo[best];
            todo[best] = todo[--left];
            g.path.push_back({(int8_t)cur, fresh});
        }
        g.pass_end.push_back((int32_t)g.path.size());
    }
}

// Channel i of a group in a chunk: window start relative to the time tile
// and the smallest relative delay.
struct Window {
    int32_t rel, bytes;
};
Window window_of(const Group &g, int i) {
    int32_t lo = INT32_MAX, hi = INT32_MIN;
    for (int k = 0; k < g.npat; ++k) {
        lo = std::min(lo, g.r[k][i]);
        hi = std::max(hi, g.r[k][i]);
    }
    Window w;
    w.rel = (g.base + lo) & ~15;
    const int32_t amax = g.base + hi - w.rel;
    // last word read: the second word of the last quad's upper half
    const int32_t words = amax / 4 + (g.quads - 1) + kSumHalf / 4 + 2;
    w.bytes = (4 * words + 15) & ~15;
    return w;
}
int32_t prog_words(const Group &g) {  // 32-bit words of a group's program
    return g.jobs * (4 + 2 * ((g.n + 1) & ~1) + 4 * 4) + 4 * g.steps;
}
int64_t raw_bytes(const Group &g) {  // delays reach 1e9 samples: a sum of windows does not fit 32 bits
    int64_t b = 0;
    for (int i = 0; i < g.n; ++i) b += window_of(g, i).bytes;
    return b;
}

// Tables of one tile; indices are relative to the tile's own arrays.
struct Tile {
    std::vector<int32_t> chunks, prog_bytes, geo, off;
    std::vector<uint32_t> prog, jobs;
    int32_t nchunks = 0, ngroups = 0;
    double clocks = 0.0;
    bool ok = true;
};

int32_t selector(int32_t byte) { return 0x3210 + 0x1111 * byte; }

// Appends one chunk: its windows' geometry, its producers' program and jobs,
// and the DM offsets of its groups.
//   program: {segments, 0, 0, 0} (what idle steps read), then per segment
//   {channels | steps << 16, row, lanes, last quad}, 8 bytes per channel {raw
//   offset of the aligned word, byte selector} (an even number), 16 per step
//   {raw offset, old selector | row << 16, new selector, lanes} and four idle
//   steps that may be prefetched.  row: where quad 0 of the pass's row would lie, in
//   units of 16 bytes (may be negative); lanes: which of the pass's quads
//   belong to the row (0: the row is not complete yet).
void emit_chunk(const sp_plan &p, int32_t d0, int cnt, const Group *gs, int ng, Tile &t) {
    const int32_t geo_first = (int32_t)(t.geo.size() / 4);
    const size_t prog_first = t.prog.size();
    int32_t words = 4, nseg = 0, nch = 0;
    for (int k = 0; k < ng; ++k) {
        words += prog_words(gs[k]);
        nseg += gs[k].jobs;
        nch += gs[k].n;
    }
    int32_t raw = 4 * words, row = 0;  // row: in quads
    const size_t job_first = t.jobs.size();
    const uint32_t use = (uint32_t)(t.nchunks / kSumSlots);
    const uint32_t slot = (uint32_t)(t.nchunks % kSumSlots) | ((use & 1u) << 2) | (use == 0 ? kSumJobFirstUse : 0u);
    t.prog.insert(t.prog.end(), {(uint32_t)nseg, 0u, 0u, 0u});
    for (int k = 0; k < ng; ++k) {
        const Group &g = gs[k];
        int32_t at[kMaxDms][kSumMaxGroup], raw_of[kSumMaxGroup], row_of[kMaxDms];
        for (int i = 0; i < g.n; ++i) {
            const Window w = window_of(g, i);
            raw_of[i] = raw;
            t.geo.insert(t.geo.end(), {w.rel, w.bytes, raw, 0});
            raw += w.bytes;
            for (int q = 0; q < g.npat; ++q) at[q][i] = g.base + g.r[q][i] - w.rel;
        }
        for (int q = 0; q < g.npat; ++q) {
            row_of[q] = row - g.qs[q];  // where quad 0 would lie
            row += g.qe[q] - g.qs[q];
        }
        for (int pass = 0, v = 0; pass < g.passes(); ++pass) {
            const int end = g.pass_end[(size_t)pass], q0 = 32 * pass;
            auto lanes = [&](int q) {  // quads of the pass that belong to pattern q's row
                const int a = std::max(0, g.qs[q] - q0), b = std::min(32, g.qe[q] - q0);
                return (uint32_t)(((b - a == 32 ? 0 : 1ull << (b - a)) - 1ull) << a);
            };
            while (v < end) {
                int e = v + 1;
                while (e < end && !g.path[(size_t)e].fresh) ++e;
                const size_t head = t.prog.size();
                const int q = g.path[(size_t)v].pat;
                t.prog.insert(t.prog.end(), {0u, (uint32_t)(row_of[q] + q0), lanes(q), (uint32_t)(g.quads - 1)});
                for (int i = 0; i < g.n; ++i) {
                    t.prog.push_back((uint32_t)(raw_of[i] + (at[q][i] & ~3)));
                    t.prog.push_back((uint32_t)selector(at[q][i] & 3));
                }
                if (g.n & 1) t.prog.insert(t.prog.end(), {0u, 0u});
                uint32_t steps = 0;
                for (int j = v + 1; j < e; ++j) {
                    const int from = g.path[(size_t)j - 1].pat, to = g.path[(size_t)j].pat;
                    for (int i = 0; i < g.n; ++i) {
                        const int32_t a0 = at[from][i], a1 = at[to][i];
                        if (a0 == a1) continue;
                        const int32_t m = std::min(a0, a1) & ~3;
                        t.prog.insert(t.prog.end(), {(uint32_t)(raw_of[i] + m),
                                                     (uint32_t)selector(a0 - m) | ((uint32_t)(row_of[to] + q0) << 16),
                                                     (uint32_t)selector(a1 - m), 0u});
                        ++steps;
                    }
                    t.prog.back() = lanes(to);  // the row is complete after its last step
                }
                t.prog[head] = (uint32_t)g.n | (steps << 16);
                t.prog.insert(t.prog.end(), 16, 0u);
                t.jobs.insert(t.jobs.end(),
                              {slot | (1u << 8), (uint32_t)((head - prog_first) / 4) | ((uint32_t)q0 << 16)});
                v = e;
            }
        }
        for (int d = 0; d < kSumDms; ++d) {
            const int dd = std::min(d, cnt - 1);  // idle slots repeat the last DM
            const int32_t b = p.delays[(size_t)(d0 + dd) * p.nchan + g.c0] - g.base;
            const int32_t flags = (d & 7) == 0 && k == ng - 1 ? kSumLastOfChunk : 0;
            t.off.push_back((16 * row_of[g.pat_of[dd]] + 4 * b) | flags);
        }
        ++t.ngroups;
    }
    t.chunks.insert(t.chunks.end(), {nch, gs[0].c0, geo_first, (int32_t)(prog_first / 4)});
    t.prog_bytes.push_back((int32_t)(t.prog.size() - prog_first) * 4);
    const uint32_t njobs = (uint32_t)(t.jobs.size() - job_first) / 2;
    t.jobs[t.jobs.size() - 2] += (uint32_t)(kSumJobArrivals - njobs) << 8;  // the last job arrives for the rest
    ++t.nchunks;
}

void build_tile(const sp_plan &p, int32_t d0, int cnt, Tile &t) {
    std::vector<Group> best(kSumMaxChunk), cand(kSumMaxChunk), open;
    open.reserve(kSumMaxChunk);
    int64_t rows = 0, raw = 0, chans = 0, jobs = 0;
    int32_t since_carry = 0;
    auto flush = [&]() {
        if (open.empty()) return;
        if (since_carry + chans > kSumCarryChannels) {  // after the chunk before this one
            for (size_t d = t.off.size() - kSumDms; d < t.off.size(); d += 8) t.off[d] |= kSumCarryAfter;
            since_carry = 0;
        }
        since_carry += (int32_t)chans;
        emit_chunk(p, d0, cnt, open.data(), (int)open.size(), t);
        t.clocks += kChunkClocks;
        open.clear();
        rows = chans = jobs = 0;
        raw = 16;
    };
    raw = 16;
    for (int32_t c0 = 0; c0 < p.nchan && t.ok; c0 += kSumMaxChunk) {
        const int32_t block = std::min(kSumMaxChunk, p.nchan - c0);
        double best_clocks = -1.0;
        int nbest = 0;
        for (int G = kSumMaxGroup; G >= 1; G >>= 1) {
            double clocks = 0.0, bytes = 0.0;
            int n = 0;
            bool fits = true;
            for (int32_t c = 0; c < block && fits; c += G) {
                Group &g = cand[n++];
                analyse(p, d0, cnt, c0 + c, std::min(G, block - c), g);
                fits = g.may_fit() && 16 + 4 * prog_words(g) + raw_bytes(g) <= kSumRawBytes &&
                       g.jobs <= kSumJobArrivals;
                clocks += group_clocks(g, cnt);
                bytes += (double)g.row_bytes();
            }
            clocks += kChunkClocks * std::max(1.0, bytes / kSumRowBytes);
            if (!fits) continue;
            if (best_clocks >= 0 && clocks >= best_clocks) break;  // smaller groups cost more still
            best_clocks = clocks;
            nbest = n;
            std::swap(best, cand);
        }
        if (best_clocks < 0) {
            t.ok = false;
            return;
        }
        for (int k = 0; k < nbest; ++k) {
            const Group &g = best[(size_t)k];
            const int64_t gr = 4 * prog_words(g) + raw_bytes(g);
            const int64_t gj = g.jobs;
            if (rows + g.row_bytes() > kSumRowBytes || raw + gr > kSumRawBytes || chans + g.n > kSumMaxChunk ||
                jobs + gj > kSumJobArrivals)
                flush();
            jobs += gj;
            rows += g.row_bytes();
            raw += gr;
            chans += g.n;
            t.clocks += group_clocks(g, cnt);
            open.push_back(g);
        }
    }
    flush();
}

}  // namespace

// SM clocks of a work item of a tile: a fixed part (set-up, first copies, output), its
// groups' modelled clocks, what a job costs besides, and the producers' time
// that consumers without trials do not cover.  Fitted to 32 plans (64 to 16384 channels,
// steps of 0.02 to 4, 9 to 64 trials a tile) with an item an SM.
static double item_clocks(const Tile &t, int32_t cnt) {
    return 38000.0 + 0.81 * t.clocks + 26.0 * (double)(t.jobs.size() / 2) +
           550.0 * t.ngroups * (kSumDms - cnt) / kSumDms;
}

// Tiles of up to kSumDms consecutive DMs, halved where a tile's delay spread
// leaves no group that fits a row slot.  SP_ELIMIT: the plan has no tables
// (too many channels for the 16-bit carries, or a table beyond int32).
static int build_tables(const sp_plan &p, SumTables &t) {
    t = SumTables();
    if (p.nchan > kSumMaxChan) return SP_ELIMIT;
    struct Span {
        int32_t first, count;
        std::vector<Tile> tiles;
        std::vector<int32_t> counts;
    };
    std::vector<Span> spans;
    for (int32_t d = 0; d < p.ndm; d += kSumDms) spans.push_back({d, std::min(kSumDms, p.ndm - d), {}, {}});
    std::atomic<size_t> next{0};
    std::atomic<bool> bad{false}, no_memory{false};
    auto work = [&]() {
        try {
            for (size_t i; (i = next.fetch_add(1)) < spans.size() && !bad;) {
                Span &s = spans[i];
                for (int32_t d = 0, want = s.count; d < s.count;) {
                    Tile tile;
                    const int32_t cnt = std::min(want, s.count - d);
                    build_tile(p, s.first + d, cnt, tile);
                    if (!tile.ok) {
                        if (cnt == 1) {  // a single DM has spread 0
                            bad = true;
                            return;
                        }
                        want = (cnt + 1) / 2;
                        continue;
                    }
                    s.tiles.push_back(std::move(tile));
                    s.counts.push_back(cnt);
                    d += cnt;
                }
            }
        } catch (...) {
            bad = no_memory = true;
        }
    };
    run_on_cores(work, (int64_t)spans.size());
    if (bad) return no_memory ? SP_ENOMEM : SP_ELIMIT;
    double clocks = 0.0;
    t.tile_most = 0.0;
    t.tile_chunk.push_back(0);
    t.tile_group.push_back(0);
    t.tile_job.push_back(0);
    for (Span &s : spans) {
        int32_t d = s.first;
        for (size_t k = 0; k < s.tiles.size(); ++k) {
            Tile &x = s.tiles[k];
            t.tile_first.push_back(d);
            t.tile_count.push_back(s.counts[k]);
            d += s.counts[k];
            if (t.geo.size() + x.geo.size() > (size_t)INT32_MAX || t.prog.size() + x.prog.size() > (size_t)INT32_MAX ||
                t.off.size() + x.off.size() > (size_t)INT32_MAX)
                return SP_ELIMIT;
            const int32_t geo0 = (int32_t)(t.geo.size() / 4), prog0 = (int32_t)(t.prog.size() / 4);
            for (int32_t c = 0; c < x.nchunks; ++c) {
                x.chunks[(size_t)4 * c + 2] += geo0;
                x.chunks[(size_t)4 * c + 3] += prog0;
            }
            t.chunks.insert(t.chunks.end(), x.chunks.begin(), x.chunks.end());
            t.prog_bytes.insert(t.prog_bytes.end(), x.prog_bytes.begin(), x.prog_bytes.end());
            t.geo.insert(t.geo.end(), x.geo.begin(), x.geo.end());
            t.prog.insert(t.prog.end(), x.prog.begin(), x.prog.end());
            t.off.insert(t.off.end(), x.off.begin(), x.off.end());
            t.jobs.insert(t.jobs.end(), x.jobs.begin(), x.jobs.end());
            t.tile_job.push_back((int32_t)(t.jobs.size() / 2));
            t.tile_chunk.push_back(t.tile_chunk.back() + x.nchunks);
            t.tile_group.push_back(t.tile_group.back() + x.ngroups);
            const double item = item_clocks(x, s.counts[k]);
            clocks += item;
            t.tile_most = std::max(t.tile_most, item);
        }
    }
    t.tile_clocks = clocks / (double)t.tile_first.size();
    return SP_OK;
}

int build_sum_tables(const sp_plan &p, SumTables &t) {
    try {
        return build_tables(p, t);
    } catch (const std::bad_alloc &) {
        return SP_ENOMEM;
    }
}

namespace {
// Direct kernel: 74 sums per SM and clock on full tiles with two items on an SM; a
// tile of few trials costs more than its share (it loads the same samples, and
// half its threads or more have no trials).  alone: an item that has its SM to itself.
constexpr double kDirectFixedClocks = 4000.0, kDirectAddsPerClock = 74.0;
constexpr double kDirectAlone = 1.32, kDirectWaves = 0.97;
double direct_item_clocks(const sp_plan &p, int32_t tile, bool alone) {
    const double full = (double)p.tile_count[(size_t)tile] / p.dm_tile;
    const double part = full > 0.5 ? 0.6 + 0.4 * full : alone ? 0.54 + 0.34 * full : 0.4 + 0.44 * full;
    return kDirectFixedClocks + part * p.dm_tile * p.time_tile * p.nchan / kDirectAddsPerClock;
}
}  // namespace

// The plan's modelled clocks of its items: shared sums and direct, average and largest.
void model_items(sp_plan &p, const SumTables &t) {
    p.sums_clocks = t.tile_clocks;
    p.sums_most = t.tile_most;
    p.direct_clocks = p.direct_most = p.direct_alone = 0.0;
    for (int32_t j = 0; j < p.ntiles; ++j) {
        const double item = direct_item_clocks(p, j, false);
        p.direct_clocks += item / p.ntiles;
        p.direct_most = std::max(p.direct_most, item);
        p.direct_alone = std::max(p.direct_alone, direct_item_clocks(p, j, true));
    }
}

// Whether a plan keeps shared-sum tables: on long inputs they beat the direct
// kernel.  DM lists whose trials share too little (coarse steps on few
// channels, random lists) stay with the direct kernel.
bool sum_tables_pay(const sp_plan &p, const SumTables &t) {
    return p.sums_clocks * (double)t.tile_first.size() / kSumTime <
           kDirectWaves * p.direct_clocks * p.ntiles / p.time_tile;
}

// Modelled clocks of one launch over these beams with either kernel.  Shared
// sums run in whole waves of an item an SM; the direct kernel's items share an
// SM as soon as they are more than the SMs.  A launch takes at least its largest item.
// Measured on 642 launches, from one item to twenty waves, of the plans that item_clocks
// was fitted to and of 45 others (trial lists of 100 to 900 pc cm^-3, 256 to 4096
// channels): nine in ten shared-sum launches take 0.97 to 1.12 of this, nine in ten
// direct launches 0.97 to 1.17.  None goes to shared sums that take longer than the
// direct kernel; 16 stay with the direct kernel and are 2 to 12 % slower.  Among them, us
// with the direct kernel and with shared sums: 4096 channels, 129 trials 1.0 apart,
// 700 samples 843, 917, 16384 samples 1101, 924; 64 channels, 512 trials 0.1 apart,
// 2048 samples 26, 41; 1024 channels, 512 trials 0.1 apart, 2048 samples 293, 172.
DedispClocks dedisp_clocks(const sp_plan *const *plans, const int64_t *n_out, int32_t nbeams, bool alike) {
    DedispClocks c;
    double sums = 0.0, direct = 0.0, direct_items = 0.0, sms = 1.0, sums_most = 0.0, direct_most = 0.0, alone = 0.0;
    for (int32_t b = 0; b < nbeams; ++b) {
        const sp_plan &p = *plans[alike ? 0 : b];
        const int64_t n = n_out[alike ? 0 : b];
        const double si = (double)sums_items(&p, n), di = (double)p.ntiles * (double)dedisp_time_tiles(&p, n);
        c.sum_items += si;
        direct_items += di;
        sums += si * p.sums_clocks;
        direct += di * p.direct_clocks;
        sums_most = std::max(sums_most, p.sums_most);
        direct_most = std::max(direct_most, p.direct_most);
        alone = std::max(alone, p.direct_alone);
        sms = p.sms;
    }
    c.sums = std::max(sums_most, std::ceil(c.sum_items / sms) * sums / c.sum_items);
    const double half_waves = std::ceil(direct_items / sms);
    if (half_waves <= 1.0) {
        c.direct = kDirectAlone * alone;
        return c;
    }
    c.direct = kDirectWaves * std::max(2.0 * direct_most, half_waves * direct / direct_items);
    if (half_waves == 3.0 || half_waves == 5.0)  // full waves, then items alone
        c.direct = std::max(c.direct, kDirectWaves * (half_waves - 1.0) * direct / direct_items + 0.9 * kDirectAlone * alone);
    return c;
}

// Whether one launch over these beams goes to the shared-sum kernel: all plans
// have tables, and the modelled clocks are fewer.
bool sums_pay(const sp_plan *const *plans, const int64_t *n_out, int32_t nbeams, bool alike) {
    for (int32_t b = 0; b < (alike ? 1 : nbeams); ++b)
        if (!plans[b]->d_sums) return false;
    const DedispClocks c = dedisp_clocks(plans, n_out, nbeams, alike);
    return c.sum_items <= INT32_MAX && c.sums < c.direct;
}

int64_t sums_items(const sp_plan *p, int64_t n_out) {
    return (int64_t)p->sums_ntiles * ((n_out + kSumTime - 1) / kSumTime);
}

// Host check of the tables against every access of the kernel and against
// the plan's delays: the number of violated conditions.
int64_t check_sum_tables(const sp_plan &p, const SumTables &t, int64_t n_out) {
    int64_t bad = 0;
    const int64_t pitch = dedisp_pitch(n_out + p.max_delay);
    const int64_t last_t0 = (n_out - 1) / kSumTime * kSumTime;
    const int32_t ntiles = (int32_t)t.tile_first.size();
    int32_t next_dm = 0;
    for (int32_t j = 0; j < ntiles; ++j) {
        const int32_t d0 = t.tile_first[j], cnt = t.tile_count[j];
        bad += (d0 != next_dm) + (cnt < 1) + (cnt > kSumDms);
        next_dm = d0 + cnt;
        int32_t g = t.tile_group[j], chan = 0, since_carry = 0, job = t.tile_job[j];
        for (int32_t k = t.tile_chunk[j]; k < t.tile_chunk[j + 1]; ++k) {
            const int32_t nch = t.chunks[(size_t)4 * k], c0 = t.chunks[(size_t)4 * k + 1];
            const int32_t *geo = &t.geo[(size_t)4 * t.chunks[(size_t)4 * k + 2]];
            const uint32_t *prog = &t.prog[(size_t)4 * t.chunks[(size_t)4 * k + 3]];
            const int32_t pbytes = t.prog_bytes[k];
            bad += (c0 != chan) + (nch < 1) + (nch > kSumMaxChunk) + (pbytes % 16 != 0) + (pbytes <= 0);
            chan += nch;
            int32_t free_from = pbytes;
            for (int32_t i = 0; i < nch; ++i) {
                const int32_t rel = geo[4 * i], bytes = geo[4 * i + 1], raw = geo[4 * i + 2];
                bad += (rel < 0) + (rel % 16 != 0) + (bytes <= 0) + (bytes % 16 != 0) + (raw % 16 != 0);
                bad += (raw < free_from) + (raw + bytes > kSumRawBytes);
                bad += (last_t0 + rel >= pitch);  // at least 16 bytes of every copy lie in the row
                free_from = raw + bytes;
            }
            // Walk the program: per pass and row, the quads stored and the
            // byte offset of each channel's first sample.
            struct Piece {
                int32_t row, q0, first, n;  // row: where quad 0 of the row would lie, in quads
                uint32_t lanes;
                std::vector<int32_t> a;     // per channel, relative to the window
            };
            std::vector<Piece> pieces;
            std::vector<int32_t> owner(kSumRowBytes / 16, -1);  // piece that stores a quad of the slot
            auto channel_of = [&](int32_t off) {
                int32_t c = -1;
                for (int32_t i = 0; i < nch; ++i)
                    if (off >= geo[4 * i + 2] && off < geo[4 * i + 2] + geo[4 * i + 1]) c = i;
                return c;
            };
            auto store = [&](const Piece &x) {
                bad += x.lanes == 0;
                for (int32_t l = 0; l < 32; ++l) {
                    if (!((x.lanes >> l) & 1u)) continue;
                    const int32_t q = x.row + x.q0 + l;
                    if (q < 0 || q >= kSumRowBytes / 16 || owner[(size_t)q] >= 0) ++bad;
                    else owner[(size_t)q] = (int32_t)pieces.size();
                }
                pieces.push_back(x);
            };
            const int32_t index = k - t.tile_chunk[j];
            const uint32_t use = (uint32_t)(index / kSumSlots);
            uint32_t arrivals = 0;
            const int32_t job0 = job;
            const uint32_t *w = prog + 4;
            for (uint32_t s = 0; s < prog[0]; ++s, ++job) {
                if (job >= t.tile_job[j + 1]) return bad + 1;
                const uint32_t x = t.jobs[(size_t)2 * job], y = t.jobs[(size_t)2 * job + 1];
                bad += (x & 3u) != (uint32_t)(index % kSumSlots) || ((x >> 2) & 1u) != (use & 1u);
                bad += ((x & kSumJobFirstUse) != 0) != (use == 0) || (x & 0xF0u) != 0 || (x >> 8) == 0;
                bad += (y & 0xFFFFu) != (uint32_t)((w - prog) / 4);
                arrivals += x >> 8;
                const int32_t n = (int32_t)(w[0] & 0xFFFFu), steps = (int32_t)(w[0] >> 16), last = (int32_t)w[3];
                const int32_t q0 = (int32_t)(y >> 16);
                Piece r{(int32_t)w[1] - q0, q0, -1, n, w[2], {}};
                bad += n < 1 || n > kSumMaxGroup || last < q0 || (q0 & 31);
                auto reads = [&](int32_t off, int32_t c) {  // words off, off + 4 of the pass's quads and both halves
                    const int32_t q = std::min(q0 + 31, last);
                    bad += c < 0 || off % 4 || off < geo[4 * c + 2] ||
                           off + 4 * q + kSumHalf + 8 > geo[4 * c + 2] + geo[4 * c + 1];
                };
                const uint32_t *e = w + 4;
                for (int32_t i = 0; i < n; ++i, e += 2) {
                    const int32_t off = (int32_t)e[0], c = channel_of(off);
                    reads(off, c);
                    if (c < 0) return bad + 1;
                    if (i == 0) r.first = c;
                    bad += c != r.first + i;
                    r.a.push_back(off - geo[4 * c + 2] + (int32_t)(e[1] & 15u));
                    bad += (int32_t)e[1] != selector((int32_t)(e[1] & 15u)) || (e[1] & 15u) > 3u;
                }
                store(r);
                if (n & 1) e += 2;
                for (int32_t i = 0; i < steps; ++i, e += 4) {
                    const int32_t off = (int32_t)e[0], c = channel_of(off);
                    reads(off, c);
                    if (c < r.first || c >= r.first + n) return bad + 1;
                    const int32_t o = (int32_t)(e[1] & 15u), q = (int32_t)(e[2] & 15u);
                    bad += o > 4 || q > 4 || (int32_t)(e[1] & 0xFFFFu) != selector(o) || (int32_t)e[2] != selector(q);
                    int32_t &a = r.a[(size_t)(c - r.first)];
                    bad += a != off - geo[4 * c + 2] + o;
                    a = off - geo[4 * c + 2] + q;
                    if (e[3]) {
                        r.row = (int32_t)(int16_t)(e[1] >> 16) - q0;
                        r.lanes = e[3];
                        store(r);
                    } else {
                        bad += i + 1 == steps;
                    }
                }
                for (int32_t i = 0; i < 16; ++i) bad += e[i] != 0;  // four idle steps that may be prefetched
                e += 16;
                bad += 4 * std::min(q0 + 31, last) + kSumHalf + 8 > kSumRawBytes;  // what they read
                w = e;
            }
            bad += (w - prog) * 4 != pbytes;
            bad += arrivals != (uint32_t)kSumJobArrivals || job - job0 < kSumMinJobs;
            // Every group: each DM's offset lies in one row whose samples
            // start at the DM's delays.
            int32_t done = 0;
            bool last = false;
            while (!last && g < t.tile_group[j + 1]) {
                const int32_t *off = &t.off[(size_t)g * kSumDms];
                last = off[0] & kSumLastOfChunk;
                int32_t n = 0;
                for (int32_t d = 0; d < kSumDms; ++d) {
                    if (d & 7) bad += (off[d] & 3) != 0;
                    else bad += (off[d] & 3) != (off[0] & 3);
                    const int32_t o = off[d] & ~3, dd = d0 + std::min(d, cnt - 1);
                    if (o < 0 || o + 4 * kSumHalf > kSumRowBytes) {
                        ++bad;
                        continue;
                    }
                    // every word it reads was stored by a piece whose samples
                    // start at the DM's delays
                    int32_t last_owner = -1;
                    for (int32_t q = o / 16; q <= (o + 4 * kSumHalf - 4) / 16; ++q) {
                        const int32_t w = owner[(size_t)q];
                        if (w < 0) {
                            ++bad;
                            break;
                        }
                        if (w == last_owner) continue;
                        last_owner = w;
                        const Piece &x = pieces[(size_t)w];
                        bad += x.first != done;
                        n = x.n;
                        for (int32_t i = 0; i < x.n; ++i)
                            bad += geo[4 * (x.first + i)] + x.a[(size_t)i] + o / 4 - 4 * x.row !=
                                   p.delays[(size_t)dd * p.nchan + c0 + x.first + i];
                    }
                }
                done += n;
                ++g;
                if (!n) break;
            }
            bad += done != nch || !last;
            since_carry += nch;
            bad += since_carry > kSumCarryChannels;
            if (g > t.tile_group[j] && (t.off[(size_t)(g - 1) * kSumDms] & kSumCarryAfter)) since_carry = 0;
        }
        bad += chan != p.nchan || g != t.tile_group[j + 1] || job != t.tile_job[j + 1];
    }
    bad += next_dm != p.ndm;
    return bad;
}

}  // namespace sp
