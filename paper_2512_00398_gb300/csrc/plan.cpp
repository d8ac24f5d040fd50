// plan.cpp -- host side of the search library: argument checking, the delay
// table (Section II-B, Eq. 1 with the cold-plasma law), the dedispersion
// tiling, workspace layout and the C ABI entry points of include/hp.h.
//
// Compiled with -ffp-contract=off: the delay table is evaluated in FP64 with
// one fixed expression order and no fused multiply-add.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "patterns.cuh"
#include "plan_internal.h"

using namespace hp;

namespace {

constexpr double kKDM = 4148.808;   // s MHz^2 pc^-1 cm^3

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
int64_t round_up64(int64_t v, int64_t a) { return (v + a - 1) / a * a; }
// bytes of sub-band partial sums held at once (chunks of DM tiles are run in
// turn when all of them would need more)
constexpr size_t kSubbandBytes = (size_t)16 << 30;

}  // namespace

namespace hp {

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// The status of a runtime call.  A failure is reported here once: the thread's last
// error is cleared, or the next launch's cudaGetLastError would report it again.
int check_cuda(cudaError_t e) {
    if (e == cudaSuccess) return HP_OK;
    (void)cudaGetLastError();
    if (e == cudaErrorMemoryAllocation) return HP_ERR_OOM;
    return HP_ERR_CUDA;
}

int plan_alloc(hp_plan* p, size_t bytes, void** out) {
    *out = nullptr;
    if (p->alloc_fn) {
        void* m = p->alloc_fn(bytes, p->alloc_ctx);
        if (!m) return HP_ERR_OOM;
        if ((uintptr_t)m & 255u) {
            p->free_fn(m, bytes, p->alloc_ctx);
            return HP_ERR_INVALID_ARG;
        }
        *out = m;
        ++p->device_allocs;
        return HP_OK;
    }
    const int rc = check_cuda(cudaMalloc(out, bytes));
    if (!rc) ++p->device_allocs;
    return rc;
}

void plan_free(hp_plan* p, void* ptr, size_t bytes) {
    if (!ptr) return;
    if (p->free_fn)
        p->free_fn(ptr, bytes, p->alloc_ctx);
    else
        cudaFree(ptr);
}

constexpr int kMaxTimedLaunches = 4096;

// Record the begin event of a stage launch; returns the pair index or -1.
int stage_begin(hp_plan* p, int stage, cudaStream_t s) {
    if (!p->timing || p->ev_used[stage] >= kMaxTimedLaunches) return -1;
    const int i = p->ev_used[stage];
    std::vector<cudaEvent_t>& v = p->ev[stage];
    while ((int)v.size() < 2 * (i + 1)) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) return -1;
        v.push_back(e);
    }
    if (cudaEventRecord(v[2 * i], s) != cudaSuccess) return -1;
    return i;
}

void stage_end(hp_plan* p, int stage, int i, cudaStream_t s) {
    if (i < 0) return;
    if (cudaEventRecord(p->ev[stage][2 * i + 1], s) == cudaSuccess) p->ev_used[stage] = i + 1;
}

// ---------------------------------------------------------------- delays
void compute_delays(hp_plan* p) {
    const int ndm = p->ndm(), nch = p->nchans;
    p->delays.assign((size_t)ndm * nch, 0);
    const double inv_top2 = 1.0 / (p->f_top * p->f_top);
    int32_t mx = 0;
    for (int d = 0; d < ndm; ++d) {
        const double dm = (double)p->dm_list[d];
        for (int c = 0; c < nch; ++c) {
            const double f = p->f_top + (double)c * p->chan_bw;
            const double sec = kKDM * dm * (1.0 / (f * f) - inv_top2);
            const int32_t v = (int32_t)std::rint(sec / p->tsamp);
            p->delays[(size_t)d * nch + c] = v;
            mx = std::max(mx, v);
        }
    }
    p->maxd = mx;
}

// ------------------------------------------------------- dedispersion tiling
// A DM tile holds up to BD consecutive trials.  For every channel the block
// stages the input row window [t0 + base, t0 + base + 4*nwords) where base =
// the channel's smallest delay over the tile rounded down to 16 bytes; trial j
// of the tile reads the words from (rel >> 2), rel = delay(c, j) - base, and
// aligns them to rel & 3 in registers.  Channels are packed into stages that
// fit the stage buffer.
struct RowGeom {
    int32_t base;
    uint32_t nwords, bbytes, smem;
};

// lo / hi: the smallest and largest delay of channel c over the tile's trials
RowGeom row_geom_span(int32_t lo, int32_t hi, int BT) {
    RowGeom g;
    g.base = lo & ~15;
    const uint32_t span = (uint32_t)(hi - g.base);
    // a trial reads words (rel >> 2) .. (rel >> 2) + BT/4
    g.nwords = (uint32_t)align_up((span >> 2) + (uint32_t)(BT / 4) + 1, 4);
    g.bbytes = 4 * g.nwords;
    g.smem = g.bbytes;
    return g;
}

// direct tables grow with the trial index, so the first and last trial bound a channel
RowGeom row_geom(const hp_plan* p, int d0, int nd, int c, int BT) {
    return row_geom_span(p->delays[(size_t)d0 * p->nchans + c],
                         p->delays[(size_t)(d0 + nd - 1) * p->nchans + c], BT);
}

// Table entries per channel pair and trial: four 32-bit words (byte offsets of
// the first word read in each channel, the PRMT selectors that align them).
uint32_t stage_table_bytes(int nchan, int BD) {
    return (uint32_t)((size_t)((nchan + 1) / 2) * BD * 4 * sizeof(uint32_t));
}

uint32_t stage_header(int nchan, int BD) {
    return (uint32_t)(align_up((size_t)nchan * sizeof(ChanDesc), 16) +
                      align_up(stage_table_bytes(nchan, BD), 16));
}

// Stages, channel descriptors and address tables of one DM tile of nd trials
// whose delay of trial j in channel c is delay(j, c); channels [0, nch) are
// cut at seg_begin[i] into segments that no stage straddles, the trials of
// segment i being written to rows seg_row[i] + j for output samples below
// nout - seg_trim[i].
template <class Delay>
int append_tile(const Delay& delay, int nd, int nch, const std::vector<int>& seg_begin,
                const std::vector<int32_t>& seg_row, const std::vector<uint32_t>& seg_trim,
                int32_t d0, const DedispConfig& C, DedispTiling* T) {
    const int BD = C.BD(), BT = C.BT();
    const uint32_t budget = (uint32_t)C.stage_bytes;
    std::vector<RowGeom> geo_all(nch);
    for (int c = 0; c < nch; ++c) {
        int32_t lo = delay(0, c), hi = lo;
        for (int j = 1; j < nd; ++j) {
            lo = std::min(lo, delay(j, c));
            hi = std::max(hi, delay(j, c));
        }
        geo_all[c] = row_geom_span(lo, hi, BT);
        if (geo_all[c].smem + stage_header(1, BD) > budget) return HP_ERR_INVALID_ARG;
    }
    TileDesc td;
    td.d0 = d0;
    td.nd = nd;
    td.stage_begin = (int32_t)T->stages.size();
    td.nstages = 0;
    const int nseg = (int)seg_begin.size();
    for (int sg = 0; sg < nseg; ++sg) {
        const int c_end = sg + 1 < nseg ? seg_begin[sg + 1] : nch;
        int c = seg_begin[sg];
        while (c < c_end) {
            int n = 0;
            uint32_t rows = 0;
            while (c + n < c_end && n < kStageMaxChans) {
                const RowGeom& g = geo_all[c + n];
                if (stage_header(n + 1, BD) + rows + g.smem > budget) break;
                rows += g.smem;
                ++n;
            }
            StageDesc sd{};
            sd.chan_begin = (uint32_t)T->chans.size();
            sd.nchan = (uint32_t)n;
            sd.addr_off = (uint32_t)align_up((size_t)n * sizeof(ChanDesc), 16);
            sd.addr_begin = (uint32_t)T->addr.size();
            sd.addr_bytes = stage_table_bytes(n, BD);
            sd.seg_row = seg_row[sg];
            sd.seg_info = (seg_trim[sg] << 1) | (c + n == c_end ? 1u : 0u);
            uint32_t off = stage_header(n, BD);
            uint32_t tx = (uint32_t)(n * sizeof(ChanDesc)) + sd.addr_bytes;
            std::vector<uint32_t> word0(n);   // per channel: byte offset of row copy 0
            for (int i = 0; i < n; ++i) {
                const RowGeom& g = geo_all[c + i];
                word0[i] = off;
                ChanDesc cd;
                cd.c = (uint32_t)(c + i);
                cd.goff = g.base;
                cd.offB = off;
                cd.nwords = g.nwords;
                T->chans.push_back(cd);
                tx += g.bbytes;
                off += g.smem;
                T->max_reach = std::max<int64_t>(T->max_reach, (int64_t)g.base + g.bbytes);
            }
            // table [pair][BD][4]: for each channel of the pair the byte offset of
            // the word trial j reads first (rel >> 2), then the two PRMT selectors
            // that take bytes rel & 3 .. 3 + (rel & 3) of each word pair
            for (int pr = 0; pr < (n + 1) / 2; ++pr) {
                for (int j = 0; j < BD; ++j) {
                    uint32_t sel[2] = {0, 0};
                    for (int e = 0; e < 2; ++e) {
                        const int i = 2 * pr + e < n ? 2 * pr + e : 2 * pr;
                        const int cc = c + i;
                        const int jj = j < nd ? j : 0;
                        const RowGeom& g = geo_all[cc];
                        const int32_t rel = delay(jj, cc) - g.base;
                        T->addr.push_back(word0[i] + 4 * ((uint32_t)rel >> 2));
                        sel[e] = 0x3210u + 0x1111u * ((uint32_t)rel & 3u);
                    }
                    T->addr.push_back(sel[0]);
                    T->addr.push_back(sel[1]);
                }
            }
            if (off > budget) return HP_ERR_INVALID_ARG;
            sd.tx_bytes = tx;
            T->stages.push_back(sd);
            td.nstages++;
            c += n;
        }
    }
    T->tiles.push_back(td);
    return HP_OK;
}

void append_tiling(std::vector<DedispTiling>& parts, DedispTiling* T) {
    size_t st = 0, ch = 0, ad = 0;
    for (const DedispTiling& q : parts) {
        st += q.stages.size();
        ch += q.chans.size();
        ad += q.addr.size();
    }
    T->stages.reserve(st);
    T->chans.reserve(ch);
    T->addr.reserve(ad);
    for (DedispTiling& q : parts) {
        for (TileDesc td : q.tiles) {
            td.stage_begin += (int32_t)T->stages.size();
            T->tiles.push_back(td);
        }
        const uint32_t c0 = (uint32_t)T->chans.size(), a0 = (uint32_t)T->addr.size();
        for (StageDesc sd : q.stages) {
            sd.chan_begin += c0;
            sd.addr_begin += a0;
            T->stages.push_back(sd);
        }
        T->chans.insert(T->chans.end(), q.chans.begin(), q.chans.end());
        T->addr.insert(T->addr.end(), q.addr.begin(), q.addr.end());
        T->max_reach = std::max(T->max_reach, q.max_reach);
        q = DedispTiling();
    }
}

// The nominal trial of the group of trial d (sub-band variant): the lower
// middle trial of the group.
int sb_nominal(const hp_plan* p, int d) {
    const int G = p->sb_group, g = d / G;
    const int len = std::min(G, p->ndm() - g * G);
    return g * G + (len - 1) / 2;
}

int build_tiling(hp_plan* p, int cfg, DedispTiling* T) {
    const DedispConfig& C = kDedispConfigs[cfg];
    const int BD = C.BD(), BT = C.BT();
    const uint32_t budget = (uint32_t)C.stage_bytes;
    const int ndm = p->ndm(), nch = p->nchans;
    T->cfg = -1;   // set once the tiling is complete
    T->BD = BD;
    T->BT = BT;
    T->tiles.clear();
    T->stages.clear();
    T->chans.clear();
    T->addr.clear();
    T->max_reach = 0;
    if (p->sb_chans > 0) {
        // Sub-band stage 1: one tile per chunk of BD groups; its trial j is the
        // nominal trial of group g0 + j, each sub-band a segment whose delays
        // are taken relative to the sub-band's first channel, written to rows
        // s * BD + j of the chunk's partial-sum block.
        if (!segmented_config(cfg)) return HP_ERR_INVALID_ARG;
        const int S = p->sb_chans;
        std::vector<int> seg_begin;
        std::vector<int32_t> seg_row;
        for (int s = 0; s < p->sb_nsub; ++s) {
            seg_begin.push_back(s * S);
            seg_row.push_back(s * BD);
        }
        for (int g0 = 0; g0 < p->sb_ngrp; g0 += BD) {
            const int nd = std::min(BD, p->sb_ngrp - g0);
            auto delay = [&](int j, int c) {
                const int32_t* row = &p->delays[(size_t)sb_nominal(p, (g0 + j) * p->sb_group) * nch];
                return row[c] - row[(c / S) * S];
            };
            // stage 2 reads a sub-band's partial sums below nout + the largest delay
            // of its first channel over the chunk's trials; stage 1 runs over
            // nout + sb_maxtop samples, so each sub-band may stop sb_maxtop - that early
            const int d_last = std::min((g0 + nd) * p->sb_group, p->ndm()) - 1;
            std::vector<uint32_t> seg_trim;
            for (int s = 0; s < p->sb_nsub; ++s)
                seg_trim.push_back((uint32_t)(p->sb_maxtop - p->delays[(size_t)d_last * nch + s * S]));
            const int rc = append_tile(delay, nd, nch, seg_begin, seg_row, seg_trim, 0, C, T);
            if (rc) return rc;
        }
        T->cfg = cfg;
        return HP_OK;
    }
    // tile boundaries: BD trials, fewer where a channel row of that many would not
    // fit a stage alone (a row only grows with the trials it serves)
    auto fits = [&](int d, int nd) {
        for (int c = nch - 1; c >= 0; --c)
            if (row_geom(p, d, nd, c, BT).smem + stage_header(1, BD) > budget) return false;
        return true;
    };
    std::vector<int> first{0};
    while (first.back() < ndm) {
        const int d0 = first.back();
        int nd = std::min(BD, ndm - d0);
        while (nd > 1 && !fits(d0, nd)) --nd;
        first.push_back(d0 + nd);
    }
    const int ntiles = (int)first.size() - 1;
    std::vector<DedispTiling> part(ntiles);   // (threads: about 0.5 ms of work each)
    std::vector<int> rcs(ntiles, HP_OK);
    const bool done = parallel_for(ntiles, (int)std::min<int64_t>((int64_t)ntiles * nch / 8192, 16), [&](int i) {
        const int32_t* base = &p->delays[(size_t)first[i] * nch];
        auto delay = [&](int j, int c) { return base[(size_t)j * nch + c]; };
        rcs[i] = append_tile(delay, first[i + 1] - first[i], nch, {0}, {first[i]}, {0u}, first[i], C, &part[i]);
    });
    if (!done) return HP_ERR_OOM;
    for (int rc : rcs)
        if (rc) return rc;
    append_tiling(part, T);
    T->cfg = cfg;
    return HP_OK;
}

// The table the dedispersion realises: the direct one, or the sub-band
// variant's effective table e(c,d) = delay(top,d) + delay(c,n) - delay(top,n)
// (top = the sub-band's first channel, n = the nominal trial of d's group),
// with the extents its two stages need.  Drops the tiling and device tables.
void apply_subband(hp_plan* p) {
    const int ndm = p->ndm(), nch = p->nchans;
    p->tiling.cfg = -1;
    int32_t mx = 0;
    if (p->sb_chans <= 0) {
        std::vector<int32_t>().swap(p->sb_eff);
        for (int32_t v : p->delays) mx = std::max(mx, v);
        p->maxd = mx;
        p->sb_nsub = p->sb_ngrp = 0;
        p->sb_maxrel = p->sb_maxtop = p->sb_spread = 0;
        return;
    }
    const int S = p->sb_chans;
    p->sb_nsub = (int32_t)ceil_div(nch, S);
    p->sb_ngrp = (int32_t)ceil_div(ndm, p->sb_group);
    p->sb_eff.assign((size_t)ndm * nch, 0);
    int32_t maxrel = 0, maxtop = 0;
    for (int d = 0; d < ndm; ++d) {
        const int32_t* at_d = &p->delays[(size_t)d * nch];
        const int32_t* at_n = &p->delays[(size_t)sb_nominal(p, d) * nch];
        int32_t* e = &p->sb_eff[(size_t)d * nch];
        for (int c = 0; c < nch; ++c) {
            const int top = (c / S) * S;
            const int32_t rel = at_n[c] - at_n[top];
            e[c] = at_d[top] + rel;
            mx = std::max(mx, e[c]);
            maxrel = std::max(maxrel, rel);
            maxtop = std::max(maxtop, at_d[top]);
        }
    }
    p->maxd = mx;
    p->sb_maxrel = maxrel;
    p->sb_maxtop = maxtop;
    // stage 2 stages, per sub-band, the window its block's trials read: the
    // spread of the sub-band's first-channel delay over the block's trials
    int32_t spread = 0;
    for (int g = 0; g < p->sb_ngrp; ++g)
        for (int d0 = g * p->sb_group; d0 < std::min((g + 1) * p->sb_group, ndm); d0 += kSubbandTrials) {
            const int d1 = std::min({d0 + kSubbandTrials, (g + 1) * p->sb_group, ndm}) - 1;
            for (int c = 0; c < nch; c += S)
                spread = std::max(spread, p->delays[(size_t)d1 * nch + c] - p->delays[(size_t)d0 * nch + c]);
        }
    p->sb_spread = spread;
}

// ------------------------------------------------------------- workspace
int64_t xt_pitch_for(int64_t nsamps) {
    int bt_max = 0;
    for (int i = 0; i < kNumDedispConfigs; ++i) bt_max = std::max(bt_max, kDedispConfigs[i].BT());
    // staged rows reach up to a tile plus a few words past the last delay
    return round_up64(nsamps + bt_max + 128, 16);
}


int64_t baseline_window(const hp_plan* p) {
    return (int64_t)std::floor(p->baseline_s / p->tsamp + 0.5);
}

int remedian_levels(int64_t win) {
    int L = 0;
    int64_t q = 1;
    while (win >= 1 && q <= win / 5) {
        q *= 5;
        ++L;
    }
    return L;
}

Layout make_layout(const hp_plan* p, int64_t nsamps, bool with_dedisp) {
    Layout L;
    L.nsamps = nsamps;
    L.nout = nsamps - p->maxd;
    const int ndm = p->ndm();
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    if (with_dedisp) {
        // stage 1 of the sub-band variant reads up to sb_maxrel samples past
        // the last sample a result uses
        L.xt_pitch = xt_pitch_for(nsamps + (p->sb_chans > 0 ? p->sb_maxrel : 0));
        L.dpitch = round_up64(L.nout, 64);
        L.xt = take((size_t)p->nchans * L.xt_pitch);
        L.D = take((size_t)ndm * L.dpitch * 4);
        if (p->fuse_levels && p->baseline_mode == 0 && p->sb_chans == 0 && L.nout > 0 &&
            remedian_levels(baseline_window(p)) >= 2) {
            L.lv2_pitch = round_up64(ceil_div(L.nout, 25), 4);
            L.lv2 = take((size_t)ndm * L.lv2_pitch * 4);
        }
        if (p->sb_chans > 0 && L.nout > 0) {
            // partial sums B of whole chunks of BD groups: nsub * BD rows per chunk
            const int64_t BD = kDedispConfigs[p->dedisp_cfg].BD();
            const int64_t nchunks = ceil_div(p->sb_ngrp, BD);
            L.sb_len = L.nout + p->sb_maxtop;
            L.sb_pitch = round_up64(L.sb_len, 64);
            const size_t chunk = (size_t)p->sb_nsub * BD * L.sb_pitch * 4;
            L.sb_chunks = (int)std::max<int64_t>(1, std::min<int64_t>(
                {nchunks, (int64_t)kMaxJobs, (int64_t)(kSubbandBytes / chunk)}));
            L.sb = take(chunk * L.sb_chunks);
        }
    }
    // RFI stage (small: per-channel counts and one int32 series of nsamps)
    {
        const int nch = p->nchans;
        const int64_t n = std::max<int64_t>(nsamps, 1);
        L.r_hist = take((size_t)nch * 256 * 4);
        L.r_med = take((size_t)nch * 4);
        L.r_spread = take((size_t)nch * 4);
        L.r_cflag = take(align_up((size_t)nch, 16));
        L.r_sflag = take((size_t)round_up64(n, 16) + 16);
        L.r_one = take(16);
        L.r_zpitch = round_up64(n, 64);
        L.r_z = take((size_t)L.r_zpitch * 4);
        const int lv = remedian_levels(baseline_window(p));
        const int q1 = std::min(lv, 5), q2 = std::min(std::max(lv - 5, 0), 5);
        int64_t p1 = 1, p2 = 1;
        for (int i = 0; i < q1; ++i) p1 *= 5;
        for (int i = 0; i < q2; ++i) p2 *= 5;
        const int64_t n1 = ceil_div(n, p1);
        L.r_lvl_pitch_a = round_up64(std::max<int64_t>(n1, 1), 4);
        L.r_lvl_pitch_b = round_up64(std::max<int64_t>(ceil_div(n1, p2), 1), 4);
        L.r_lvl_a = take((size_t)L.r_lvl_pitch_a * 4);
        L.r_lvl_b = take((size_t)L.r_lvl_pitch_b * 4);
        L.r_mean_pitch = ceil_div(n, 32) + 1;
        L.r_mean = take(p->baseline_mode == 1 ? (size_t)L.r_mean_pitch * 8 : 0);
        L.r_zhist = take((size_t)kHistBins * 4);
        L.r_bucket = take(8);
        L.r_rank = take(8);
        L.r_mad = take(8);
        L.r_sigma = take(8);
        L.r_tint = take(8);
        L.r_y = take(p->baseline_mode == 1 ? (size_t)L.r_zpitch * 4 : 0);
    }
    L.search_begin = off;
    // y = D - b: written over the plan's own dedispersed series in median mode
    // (whose baseline reads only the remedian knots); a separate array in mean
    // mode (the moving window reads D around each sample) and for a caller's
    // series (hp_detect leaves it unchanged)
    L.y_in_D = with_dedisp && p->baseline_mode == 0;
    if (!L.y_in_D) {
        L.ypitch = round_up64(std::max<int64_t>(L.nout, 1), 64);
        L.y = take((size_t)ndm * L.ypitch * 4);
    }
    // remedian passes of up to five levels: pass 1 writes buffer a, pass 2
    // buffer b, later passes alternate (each pass shrinks the series)
    const int levels = remedian_levels(baseline_window(p));
    const int q1 = std::min(levels, 5), q2 = std::min(std::max(levels - 5, 0), 5);
    int64_t p1 = 1, p2 = 1;
    for (int i = 0; i < q1; ++i) p1 *= 5;
    for (int i = 0; i < q2; ++i) p2 *= 5;
    const int64_t n1 = ceil_div(std::max<int64_t>(L.nout, 1), p1);
    L.lvl_pitch_a = round_up64(std::max<int64_t>(n1, 1), 4);
    L.lvl_pitch_b = round_up64(std::max<int64_t>(ceil_div(n1, p2), 1), 4);
    L.lvl_a = take((size_t)ndm * L.lvl_pitch_a * 4);
    L.lvl_b = take((size_t)ndm * L.lvl_pitch_b * 4);
    L.mean_pitch = ceil_div(std::max<int64_t>(L.nout, 1), 32) + 1;
    L.mean = take(p->baseline_mode == 1 ? (size_t)ndm * L.mean_pitch * 8 : 0);
    L.hist = take((size_t)ndm * kHistBins * 4);
    L.rbucket = take((size_t)ndm * 4);
    L.rrank = take((size_t)ndm * 8);
    L.mad = take((size_t)ndm * 8);
    L.ybound = take((size_t)ndm * 8);
    L.sigma = take((size_t)ndm * 8);
    L.tint = take((size_t)ndm * p->nw() * 8);
    if (p->decimate > 0) {
        // the distinct block sizes q = W / R of the decimated widths, ascending,
        // and one scrunched series per q
        std::vector<int32_t> qs;
        for (int32_t W : p->widths)
            if (W > p->decimate && W % p->decimate == 0) qs.push_back(W / p->decimate);
        std::sort(qs.begin(), qs.end());
        qs.erase(std::unique(qs.begin(), qs.end()), qs.end());
        L.ndec = (int)qs.size();
        size_t bytes = 0;
        for (int l = 0; l < L.ndec; ++l) {
            L.dec_q[l] = qs[l];
            L.dec_pitch[l] = round_up64(std::max<int64_t>(L.nout / qs[l], 1), 64);
            L.dec_off[l] = (int64_t)(bytes / 4);
            bytes += (size_t)ndm * L.dec_pitch[l] * 4;
        }
        if (L.ndec > 0) {
            L.ydec = take(bytes);
            L.tint_lv = take((size_t)L.ndec * ndm * p->nw() * 8);
            L.widths_lv = take((size_t)L.ndec * p->nw() * 4);
        }
    }
    if (p->width_sigma) {
        const size_t pairs = (size_t)ndm * p->nw();
        L.whist = take(pairs * 2 * 4096 * 4);
        L.wstate = take(pairs * sizeof(WsigState));
        L.wmad = take(pairs * 8);
        L.sigw = take(pairs * 8);
    }
    L.tails = take((size_t)kTailCap * sizeof(TailRec));
    L.tcount = take(8);
    const size_t cap = (size_t)p->raw_capacity;
    // the sort works on whole chunks: key/value scratch is padded to a chunk multiple
    const size_t cap_pad = align_up(cap, (size_t)kSortChunk);
    L.raw = take(cap * sizeof(hp_raw_cand));
    L.raw_count = take(8);
    L.keys0 = take(cap_pad * 8);
    L.keys1 = take(cap_pad * 8);
    L.vals0 = take(cap_pad * 8);
    L.vals1 = take(cap_pad * 8);
    L.parent = take(cap * 4);
    L.best = take(cap * 8);
    L.rep = take(cap * 4);
    L.members = take(cap * 4);
    L.dmlo = take(cap * 4);
    L.dmhi = take(cap * 4);
    L.tlo = take(cap * 8);
    L.thi = take(cap * 8);
    L.scan = take(cap * 4);
    L.bsums = take((cap / 1024 + 2) * 4);
    L.nclamp = take(8);
    L.tstart = take(((int64_t)p->ndm() + 1) * 8);
    L.total = off;
    return L;
}

// Constant tables from (pageable) host vectors, on the device when finish() returns:
// any stream may launch the kernel that reads them.  The copies run on the call's own
// stream, after whatever still uses memory that a stream-ordered allocator hands out
// again.  (cudaMemcpy alone may return while its last piece is still on the way, on a
// stream that non-blocking ones do not wait for.)
struct TableUpload {
    cudaStream_t s;
    int rc = HP_OK;
    explicit TableUpload(cudaStream_t stream) : s(stream) {
        // under capture the legacy stream, as nothing may wait for s
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        rc = check_cuda(cudaStreamIsCapturing(s, &cap));
        if (cap != cudaStreamCaptureStatusNone) s = cudaStreamLegacy;
    }
    void put(void* dst, const void* src, size_t bytes) {
        if (!rc && bytes) rc = check_cuda(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s));
    }
    int finish() {
        const int e = check_cuda(cudaStreamSynchronize(s));
        return rc ? rc : e;
    }
};

int ensure_device_tables(hp_plan* p, cudaStream_t s) {
    const int64_t sb_key = p->sb_chans > 0 ? ((int64_t)p->sb_chans << 32) | p->sb_group : 0;
    if (p->tables && p->tables_cfg == p->dedisp_cfg && p->tables_sb == sb_key) return HP_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HP_ERR_CUDA;
    if (p->tiling.cfg != p->dedisp_cfg) {
        int rc = build_tiling(p, p->dedisp_cfg, &p->tiling);
        if (rc) return rc;
    }
    if (cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return HP_ERR_CUDA;
    const DedispTiling& T = p->tiling;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    const size_t o_status = take(256);
    const size_t o_tiles = take(T.tiles.size() * sizeof(TileDesc));
    const size_t o_stages = take(T.stages.size() * sizeof(StageDesc));
    const size_t o_chans = take(T.chans.size() * sizeof(ChanDesc));
    const size_t o_addr = take(T.addr.size() * sizeof(uint32_t));
    const size_t o_widths = take(p->widths.size() * sizeof(int32_t));
    // sub-band variant: delay of every sub-band's first channel per trial
    std::vector<int32_t> sbtop;
    if (p->sb_chans > 0) {
        sbtop.resize((size_t)p->ndm() * p->sb_nsub);
        for (int d = 0; d < p->ndm(); ++d)
            for (int sb = 0; sb < p->sb_nsub; ++sb)
                sbtop[(size_t)d * p->sb_nsub + sb] =
                    p->delays[(size_t)d * p->nchans + (size_t)sb * p->sb_chans];
    }
    const size_t o_sbtop = take(sbtop.size() * sizeof(int32_t));
    const size_t total = off;
    int prev_status = p->pending_status;
    p->pending_status = 0;
    if (p->tables) {
        if (p->status) cudaMemcpy(&prev_status, p->status, sizeof(int), cudaMemcpyDeviceToHost);
        cudaDeviceSynchronize();
        plan_free(p, p->tables, p->tables_bytes);
        p->tables = nullptr;
    }
    void* mem = nullptr;
    int rc = plan_alloc(p, total, &mem);
    if (rc) return rc;
    uint8_t* b = (uint8_t*)mem;
    TableUpload up(s);
    up.put(b + o_status, &prev_status, sizeof(int));
    up.put(b + o_tiles, T.tiles.data(), T.tiles.size() * sizeof(TileDesc));
    up.put(b + o_stages, T.stages.data(), T.stages.size() * sizeof(StageDesc));
    up.put(b + o_chans, T.chans.data(), T.chans.size() * sizeof(ChanDesc));
    up.put(b + o_addr, T.addr.data(), T.addr.size() * sizeof(uint32_t));
    up.put(b + o_widths, p->widths.data(), p->widths.size() * sizeof(int32_t));
    up.put(b + o_sbtop, sbtop.data(), sbtop.size() * sizeof(int32_t));
    rc = up.finish();
    if (rc) {
        plan_free(p, mem, total);
        return rc;
    }
    p->tables = mem;
    p->tables_bytes = total;
    p->tables_cfg = p->dedisp_cfg;
    p->tables_sb = sb_key;
    p->device = dev;
    p->status = (int*)(b + o_status);
    p->d_tiles = (const TileDesc*)(b + o_tiles);
    p->d_stages = (const StageDesc*)(b + o_stages);
    p->d_chans = (const ChanDesc*)(b + o_chans);
    p->d_addr = (const uint32_t*)(b + o_addr);
    p->d_widths = (int32_t*)(b + o_widths);
    p->d_sbtop = sbtop.empty() ? nullptr : (const int32_t*)(b + o_sbtop);
    return HP_OK;
}

int ensure_workspace(hp_plan* p, size_t need, uint8_t** base) {
    if (p->ws_user) {
        if (p->ws_user_bytes < need) return HP_ERR_OOM;
        *base = (uint8_t*)p->ws_user;
        return HP_OK;
    }
    if (p->ws_own_bytes < need) {
        if (p->ws_own) {
            cudaDeviceSynchronize();
            plan_free(p, p->ws_own, p->ws_own_bytes);
            p->ws_own = nullptr;
            p->ws_own_bytes = 0;
        }
        int rc = plan_alloc(p, need, &p->ws_own);
        if (rc) return rc;
        p->ws_own_bytes = need;
    }
    *base = (uint8_t*)p->ws_own;
    return HP_OK;
}

// Every staged row of the last time tile stays inside the transposed row (the
// copies never read past the buffer).
bool reach_ok(const hp_plan* p, int64_t nout, int64_t xt_pitch) {
    const int64_t last_t0 = (ceil_div(nout, p->tiling.BT) - 1) * (int64_t)p->tiling.BT;
    return last_t0 + p->tiling.max_reach <= xt_pitch;
}

// How a launch of `total` pattern-row blocks is divided: the tiles of the last *cols of the
// last input's ntt time columns (0: none) are shared by *parts blocks each, where that
// takes the fewest waves, of tiles alike.  A block takes a tile's channels one after
// another for up to a millisecond, and one block fits an SM: 320 blocks (375 trials, four
// gulps) on 152 SMs took three such waves where 2.1 would do.  A part takes 1 / parts of a wave and
// `fixed` more to fill its pipeline and to add its sums to the output; a
// gain of less than 4% or 0.15 waves is left, as the kernel that takes parts of tiles is
// 1 to 2% slower and tiles of high delays take longer than the others.  Measured, whole
// tiles and parts by this rule, 4096 channels: 1500 trials x 9215 samples (2.07 waves)
// 2.12 and 1.58 ms; 375 x 83968 (4.32) 4.06 and 3.64; 1500 x 129 000 (26.1) 12.80 and
// 12.61; 750 x 8192 (0.84) 0.833, 0.869 split against the rule.
void pattern_waves(const hp_plan* p, const PatternCost& cost, int64_t total, int ntt, int* cols, int* parts) {
    *cols = 0;
    *parts = 1;
    const int64_t sms = p->sm_count, nq = ceil_div(p->ndm(), kPatBD);
    const double best = (double)ceil_div(total, sms);
    double limit = best - std::max(0.04 * best, 0.15);
    const double fixed = 20000.0 * (double)nq / cost.sum;
    const int max_parts = std::min(16, p->nchans / 64);
    for (int c = 1; c <= std::min(ntt, 24) && c * nq <= 2 * sms; ++c)
        for (int k = 2; k <= max_parts; ++k) {
            const int64_t whole = total - c * nq, waves = ceil_div(whole, sms);
            const double unit = 1.0 / k + fixed;
            // parts that fit the idle SMs of the last whole wave, then waves of parts
            const int64_t rest = c * nq * k - (waves * sms - whole) * (int64_t)(1.0 / unit);
            const double t = (double)waves + (rest > 0 ? (double)ceil_div(rest, sms) * unit : 0.0);
            if (t < limit) {
                limit = t;
                *cols = c;
                *parts = k;
            }
        }
}

// To start a block and fill and drain its pipeline, from a launch's second wave on (either
// kernel; the first is part of every launch).
constexpr double kBlockCycles = 12000.0;

// Estimated SM cycles of a launch so divided.  Tiles of high delays have more patterns, up
// to ten times the cycles of the first ones on a grid that widens with the DM, and come
// last: a launch ends with some of those, whatever the average.  Zeroing the output for
// the parts is a launch more.  Fitted, as the other estimates here, to 4837 launches
// (100-4096 channels, 20-1500 trials, 1000-150 000 samples, even and widening grids) and
// 20 555 divisions of them: measured / estimated 0.96-1.03 for whole tiles and 0.93-1.10
// for parts (5th to 95th of 100; no better with the blocks' order simulated).
double pattern_cycles(const hp_plan* p, const PatternCost& cost, int64_t total, int cols, int parts) {
    const double sms = p->sm_count, nq = (double)ceil_div(p->ndm(), kPatBD);
    auto waves = [&](double n, double each, double last) {
        const double w = std::ceil(n / sms);
        return w <= 1 ? last : std::max(w * each, std::min((w - 1) * each + last, n * each / sms + 0.7 * last));
    };
    const double tile = cost.sum / nq + kBlockCycles, last = cost.top + kBlockCycles;
    if (cols == 0) return waves((double)total, tile, last) - kBlockCycles;
    const double n = cols * nq * parts, whole = (double)total - cols * nq;
    const double part = 1.04 * cost.sum / nq / parts + 28000.0, end = 1.04 * cost.top / parts + 28000.0;
    // (the parts fill SMs from the last whole wave on)
    return 10000.0 + (whole <= 0 ? waves(n, part, end)
                                 : std::max(1.02 * waves(whole, tile, last),
                                            (1.02 * whole * tile + n * part) / sms + 0.7 * end));
}

// Is a launch of njobs inputs (nout[j] samples) faster with pattern rows of tiles that
// cost that much?  Both kernels keep one block per SM, so the one whose last wave ends first,
// by the estimated cycles of its blocks: the pattern rows' larger tiles (24 trials x 2048
// samples against 15 x 2176) lose on short inputs, where a wave is nearly empty, and
// where the last tiles share little, although they take fewer cycles per sum; sharing
// tiles among blocks (pattern_waves) makes up for that on many short inputs: 4096 channels, 375
// trials, 4000 samples 0.833 ms by byte rows, 0.256 by parts of pattern rows; 2048
// channels, 200 trials, 8192 samples 0.421 and 0.160.  (Near ties of parts, whose
// estimate is the rougher one, go to the byte rows, those of whole tiles to the pattern
// rows: these lose less beside other files' searches -- a batch of four files with one
// such tie 18.44 and 18.71 ms.)  On 2500 launches like those above, but others, this takes
// 0.60 of the byte rows' time (geometric mean), and 11 are more than 3% slower than byte
// rows, up to 1.2 times (256 channels, parts); by the average tile they were 102, up to 2.2
// times (512 channels, 240 trials to DM 312, 8000 samples: 0.194 and 0.123 ms).  The tables make the plan's first call longer: with both kernels' it takes
// 1.2 ms more than a later one on 1024 channels x 24 trials, 3.3 on 1024 x 400, 22 on
// 4096 x 1500 (with the byte rows' alone, built by one thread, 0.35, 3.5 and 57).
bool patterns_pay(const hp_plan* p, const PatternCost& cost, const int64_t* nout, int njobs) {
    // the default tile shape of direct dedispersion, without fused remedian levels
    if (p->dedisp_cfg != kDefaultDedispConfig || p->sb_chans > 0 || p->fuse_levels) return false;
    if (cost.sum <= 0 || njobs < 1) return false;
    const DedispTiling& T = p->tiling;
    int64_t qcols = 0, tcols = 0;
    for (int j = 0; j < njobs; ++j) {
        if (nout[j] <= 0) return false;
        qcols += ceil_div(nout[j], kPatBT);
        tcols += ceil_div(nout[j], T.BT);
    }
    const double t = (double)ceil_div(tcols * (int64_t)T.tiles.size(), p->sm_count) *
                     (byte_row_cycles((double)T.BD * p->nchans * T.BT) + kBlockCycles) - kBlockCycles;
    const int64_t total = qcols * ceil_div(p->ndm(), kPatBD);
    int cols, parts;
    pattern_waves(p, cost, total, (int)ceil_div(nout[njobs - 1], kPatBT), &cols, &parts);
    return pattern_cycles(p, cost, total, cols, parts) * (cols > 0 ? 1.03 : 0.98) < t;
}

bool use_patterns(const hp_plan* p, const int64_t* nout, const int64_t* xt_pitch, int njobs) {
    const DedispTiling& Q = p->ptiling;
    if (!p->ptables) return false;
    for (int j = 0; j < njobs; ++j)
        if ((ceil_div(nout[j], Q.BT) - 1) * Q.BT + Q.max_reach > xt_pitch[j]) return false;
    return patterns_pay(p, Q.cost, nout, njobs);
}

// While it lives, this thread's allocations and copies are allowed beside another
// stream's capture, which would otherwise (in the global mode, torch's default) be
// invalidated by them.
struct BesideCaptures {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    BesideCaptures() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
    ~BesideCaptures() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
};

int prepare_patterns(hp_plan* p, int64_t nout, int njobs, cudaStream_t s) {
    if (p->ptables || p->pat_estimate.sum < 0 || p->dedisp_cfg != kDefaultDedispConfig ||
        p->sb_chans > 0 || p->fuse_levels)
        return HP_OK;
    if (p->pat_estimate.sum == 0) {
        // (of 1250 plans 98 in 100 come out 4% above to 5% below their tables' own cost: a
        // near tie builds them and is decided by that)
        p->pat_estimate = estimate_patterns(p);
        p->pat_estimate.sum *= 0.96;
        p->pat_estimate.top *= 0.96;
    }
    int64_t nouts[kMaxJobs];
    std::fill_n(nouts, kMaxJobs, nout);
    if (!patterns_pay(p, p->pat_estimate, nouts, std::min(njobs, kMaxJobs))) return HP_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (check_cuda(cudaStreamIsCapturing(s, &cap)) || cap != cudaStreamCaptureStatusNone)
        return HP_OK;
    DedispTiling& Q = p->ptiling;
    if (!Q.pattern && !build_patterns(p, &Q)) {
        p->pat_estimate.sum = -1;
        return HP_OK;
    }
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    const size_t o_tiles = take(Q.tiles.size() * sizeof(TileDesc));
    const size_t o_stages = take(Q.stages.size() * sizeof(StageDesc));
    const size_t o_chans = take(Q.chans.size() * sizeof(ChanDesc));
    const size_t o_addr = take(Q.addr.size() * sizeof(uint32_t));
    const BesideCaptures beside;   // (a later call than the plan's first may come here)
    void* mem = nullptr;
    int rc = plan_alloc(p, off, &mem);
    if (rc) {               // no room: the byte rows run, from now on (no call asks again)
        Q = DedispTiling();
        p->pat_estimate.sum = -1;
        return HP_OK;
    }
    uint8_t* b = (uint8_t*)mem;
    TableUpload up(s);
    up.put(b + o_tiles, Q.tiles.data(), Q.tiles.size() * sizeof(TileDesc));
    up.put(b + o_stages, Q.stages.data(), Q.stages.size() * sizeof(StageDesc));
    up.put(b + o_chans, Q.chans.data(), Q.chans.size() * sizeof(ChanDesc));
    up.put(b + o_addr, Q.addr.data(), Q.addr.size() * sizeof(uint32_t));
    rc = up.finish();
    if (rc) {
        plan_free(p, mem, off);
        return rc;
    }
    // (the host needs only the tile list, the extents and the estimate from now on)
    std::vector<StageDesc>().swap(Q.stages);
    std::vector<ChanDesc>().swap(Q.chans);
    std::vector<uint32_t>().swap(Q.addr);
    p->ptables = mem;
    p->ptables_bytes = off;
    p->d_ptiles = (const TileDesc*)(b + o_tiles);
    p->d_pstages = (const StageDesc*)(b + o_stages);
    p->d_pchans = (const ChanDesc*)(b + o_chans);
    p->d_paddr = (const uint32_t*)(b + o_addr);
    return HP_OK;
}

void drop_patterns(hp_plan* p) {
    cudaDeviceSynchronize();
    plan_free(p, p->ptables, p->ptables_bytes);
    p->ptables = nullptr;
    p->ptables_bytes = 0;
    p->ptiling = DedispTiling();
    p->pat_estimate.sum = -1;
}

DedispJob make_job(const hp_plan* p, const uint8_t* xt, int64_t xt_pitch, int32_t* out,
                   int64_t out_pitch, int64_t nout, bool pat) {
    DedispJob J;
    const DedispTiling& T = pat ? p->ptiling : p->tiling;
    J.xt = xt;
    J.xt_pitch = xt_pitch;
    J.out = out;
    J.out_pitch = out_pitch;
    J.nout = nout;
    J.ntt = (int32_t)ceil_div(nout, T.BT);
    J.ndt = (int32_t)T.tiles.size();
    if (!pat && !reach_ok(p, nout, xt_pitch)) J.ntt = J.ndt = 0;   // callers report the error
    J.tiles = pat ? p->d_ptiles : p->d_tiles;
    J.stages = pat ? p->d_pstages : p->d_stages;
    J.chans = pat ? p->d_pchans : p->d_chans;
    J.addr = pat ? p->d_paddr : p->d_addr;
    J.lv = nullptr;
    J.lv_pitch = 0;
    J.pattern = pat ? 1 : 0;
    return J;
}

// Split the last time tiles of a launch of pattern-row jobs of plan p over several
// blocks each (plan_internal.h).
int split_tail(const hp_plan* p, DedispBatch* b, cudaStream_t s) {
    if (b->njobs < 1 || b->njobs >= kMaxJobs) return HP_OK;
    for (int j = 0; j < b->njobs; ++j)
        if (b->jobs[j].pattern != 1) return HP_OK;
    DedispJob& J = b->jobs[b->njobs - 1];
    const int64_t nq = J.ndt;
    int cols = 0, parts = 1;
    pattern_waves(p, p->ptiling.cost, b->prefix[b->njobs], J.ntt, &cols, &parts);
    if (cols == 0) return HP_OK;
    DedispJob& Q = b->jobs[b->njobs];
    Q = J;
    const int64_t t1 = (int64_t)(J.ntt - cols) * kPatBT;
    Q.xt += t1;
    Q.out += t1;
    Q.nout -= t1;
    Q.ntt = cols;
    Q.pattern = parts;
    J.nout = t1;
    J.ntt -= cols;
    b->prefix[b->njobs] -= (int64_t)cols * nq;
    b->prefix[b->njobs + 1] = b->prefix[b->njobs] + (int64_t)cols * nq * parts;
    ++b->njobs;
    return check_cuda(cudaMemset2DAsync(Q.out, (size_t)Q.out_pitch * 4, 0, (size_t)Q.nout * 4,
                                        (size_t)p->ndm(), s));
}

int launched_kernel(const DedispBatch& b) {
    int64_t k = 0;
    for (int j = 0; j < b.njobs; ++j) k = std::max(k, b.jobs[j].pattern);
    return (int)k;
}

// The dedispersion of the plan's own series also writes the second remedian
// level (median baseline with at least two levels, direct dedispersion: the
// layout holds the buffer only then), and the search starts from it.
void fuse_levels(DedispJob& J, const Layout& L, uint8_t* ws) {
    if (L.lv2_pitch > 0) {
        J.lv = (int32_t*)(ws + L.lv2);
        J.lv_pitch = L.lv2_pitch;
    }
}

void fuse_levels(SearchArgs& a, const Layout& L, uint8_t* ws, int cfg) {
    if (L.lv2_pitch > 0) {
        a.lv2 = (int32_t*)(ws + L.lv2);
        a.lv2_pitch = L.lv2_pitch;
        a.lv2_bt = kDedispConfigs[cfg].BT();
    }
}

// Stages 1 and 2 of the sub-band variant on the transposed input: per chunk
// set, one segmented byte-row launch (partial sums of every sub-band at the
// nominal trials of BD groups per chunk) and one sum launch (per trial, the
// shifted partial sums of every sub-band).
int run_subband(hp_plan* p, const Layout& L, uint8_t* ws, int32_t* out, int64_t out_pitch,
                cudaStream_t s) {
    const DedispTiling& T = p->tiling;
    const int nchunks = (int)T.tiles.size();
    const int64_t rows = (int64_t)p->sb_nsub * T.BD;     // partial-sum rows per chunk
    int32_t* B = (int32_t*)(ws + L.sb);
    if (!reach_ok(p, L.sb_len, L.xt_pitch)) return HP_ERR_INVALID_ARG;
    for (int c0 = 0; c0 < nchunks; c0 += L.sb_chunks) {
        const int n = std::min(L.sb_chunks, nchunks - c0);
        DedispBatch db;
        std::memset(&db, 0, sizeof(db));
        db.njobs = n;
        for (int k = 0; k < n; ++k) {
            DedispJob J = make_job(p, ws + L.xt, L.xt_pitch, B + (size_t)k * rows * L.sb_pitch,
                                   L.sb_pitch, L.sb_len, false);
            J.tiles = p->d_tiles + (c0 + k);
            J.ndt = 1;
            db.jobs[k] = J;
            db.prefix[k + 1] = db.prefix[k] + (int64_t)J.ntt * J.ndt;
        }
        int ti = stage_begin(p, HP_STAGE_DEDISP, s);
        int rc = check_cuda(launch_dedisp_segmented(p->dedisp_cfg, db, p->status, p->timeout_ns, s));
        stage_end(p, HP_STAGE_DEDISP, ti, s);
        if (rc) return rc;
        ++p->launches;
        p->last_kernel = 0;
        SubbandArgs a;
        a.B = B;
        a.bpitch = L.sb_pitch;
        a.top = p->d_sbtop;
        a.nsub = p->sb_nsub;
        a.G = p->sb_group;
        a.gchunk = T.BD;
        a.c0 = c0;
        a.g_begin = c0 * T.BD;
        a.g_end = std::min((c0 + n) * T.BD, p->sb_ngrp);
        a.ndm = p->ndm();
        a.win_cap = (int32_t)align_up((size_t)kSubbandTile + p->sb_spread + 8, 4);
        a.out = out;
        a.out_pitch = out_pitch;
        a.nout = L.nout;
        a.status = p->status;
        a.timeout_ns = p->timeout_ns;
        ti = stage_begin(p, HP_STAGE_SUBBAND_SUM, s);
        rc = check_cuda(launch_subband_sum(a, s));
        stage_end(p, HP_STAGE_SUBBAND_SUM, ti, s);
        if (rc) return rc;
        ++p->launches;
    }
    return HP_OK;
}

// Transpose, optional RFI mitigation, dedispersion (direct or sub-band) of one
// input into out[ndm][out_pitch].
int run_dedisp(hp_plan* p, const uint8_t* fb, int64_t nsamps, const Layout& L, uint8_t* ws,
               int32_t* out, int64_t out_pitch, cudaStream_t s, bool with_rfi, bool own_series) {
    uint8_t* xt = ws + L.xt;
    const int64_t xt_pitch = L.xt_pitch;
    const int64_t nout = nsamps - p->maxd;
    int ti = stage_begin(p, HP_STAGE_TRANSPOSE, s);
    int rc = check_cuda(launch_transpose(fb, nsamps, p->nchans, xt, xt_pitch, s));
    stage_end(p, HP_STAGE_TRANSPOSE, ti, s);
    if (rc) return rc;
    ++p->launches;
    if (p->rfi && with_rfi) {
        const RfiArgs r = make_rfi_args(p, L, ws, fb, xt, xt_pitch, nsamps, nullptr);
        ti = stage_begin(p, HP_STAGE_RFI, s);
        rc = check_cuda(launch_rfi(r, s, &p->launches));
        stage_end(p, HP_STAGE_RFI, ti, s);
        if (rc) return rc;
    }
    if (p->sb_chans > 0) return run_subband(p, L, ws, out, out_pitch, s);
    rc = prepare_patterns(p, nout, 1, s);
    if (rc) return rc;
    DedispBatch B;   // copied into the kernel parameters at launch
    std::memset(&B, 0, sizeof(B));
    B.njobs = 1;
    if (!reach_ok(p, nout, xt_pitch)) return HP_ERR_INVALID_ARG;
    B.jobs[0] = make_job(p, xt, xt_pitch, out, out_pitch, nout, use_patterns(p, &nout, &xt_pitch, 1));
    if (own_series) fuse_levels(B.jobs[0], L, ws);
    B.prefix[0] = 0;
    B.prefix[1] = (int64_t)B.jobs[0].ntt * B.jobs[0].ndt;
    ti = stage_begin(p, HP_STAGE_DEDISP, s);
    rc = split_tail(p, &B, s);
    if (!rc) rc = check_cuda(launch_dedisp(p->dedisp_cfg, B, p->status, p->timeout_ns, s));
    stage_end(p, HP_STAGE_DEDISP, ti, s);
    if (!rc) {
        ++p->launches;
        p->last_kernel = launched_kernel(B);
    }
    return rc;
}

int validate_search_input(const hp_plan* p, const void* ptr, int64_t nsamps) {
    if (!p || !ptr) return HP_ERR_INVALID_ARG;
    if (nsamps <= 0 || nsamps >= kMaxSamples) return HP_ERR_INVALID_ARG;
    if (nsamps <= (int64_t)p->maxd + p->wmax) return HP_ERR_NSAMPS_TOO_SHORT;
    return HP_OK;
}

SearchArgs make_search_args(hp_plan* p, const Layout& L, uint8_t* ws, const int32_t* D,
                            int64_t pitch, int64_t nout, hp_raw_cand* raw, int64_t raw_cap,
                            int64_t* raw_count) {
    SearchArgs a;
    a.D = D;
    a.pitch = pitch;
    a.nout = nout;
    a.ndm = p->ndm();
    a.nw = p->nw();
    a.widths = p->d_widths;
    a.wmax = p->wmax;
    a.thr = p->thr;
    a.baseline_mode = p->baseline_mode;
    a.win = baseline_window(p);
    a.levels = remedian_levels(a.win);
    a.lv2 = nullptr;
    a.lv2_pitch = 0;
    a.lv2_bt = 0;
    a.lvl_a = (int32_t*)(ws + L.lvl_a);
    a.lvl_b = (int32_t*)(ws + L.lvl_b);
    a.lvl_pitch_a = L.lvl_pitch_a;
    a.lvl_pitch_b = L.lvl_pitch_b;
    a.mean_pre = (int64_t*)(ws + L.mean);
    a.mean_pitch = L.mean_pitch;
    a.hist = (uint32_t*)(ws + L.hist);
    a.refine_bucket = (int32_t*)(ws + L.rbucket);
    a.refine_rank = (int64_t*)(ws + L.rrank);
    a.mad = (int64_t*)(ws + L.mad);
    a.ybound = (int64_t*)(ws + L.ybound);
    a.ybound_w = p->wmax;
    a.sigma = (double*)(ws + L.sigma);
    a.tint = (int64_t*)(ws + L.tint);
    a.raw = raw;
    a.raw_cap = raw_cap;
    a.raw_count = raw_count;
    a.tails = (TailRec*)(ws + L.tails);
    a.tail_cap = kTailCap;
    a.tail_count = (int64_t*)(ws + L.tcount);
    a.status = p->status;
    if (L.y_in_D) {
        a.Y = const_cast<int32_t*>(D);
        a.ypitch = pitch;
    } else {
        a.Y = (int32_t*)(ws + L.y);
        a.ypitch = L.ypitch;
    }
    a.nwin = nout;
    a.carry_in = nullptr;
    a.carry_out = nullptr;
    a.t_offset = 0;
    a.stats_only = 0;
    a.sample_mul = 1;
    a.decimate = p->decimate;
    a.ndec = L.ndec;
    for (int l = 0; l < L.ndec; ++l) {
        a.dec_q[l] = L.dec_q[l];
        a.dec_off[l] = L.dec_off[l];
        a.dec_pitch[l] = L.dec_pitch[l];
    }
    a.ydec = L.ndec > 0 ? (int32_t*)(ws + L.ydec) : nullptr;
    a.tint_lv = L.ndec > 0 ? (int64_t*)(ws + L.tint_lv) : nullptr;
    a.widths_lv = L.ndec > 0 ? (int32_t*)(ws + L.widths_lv) : nullptr;
    a.width_sigma = p->width_sigma ? 1 : 0;
    a.whist = p->width_sigma ? (uint32_t*)(ws + L.whist) : nullptr;
    a.wstate = p->width_sigma ? (WsigState*)(ws + L.wstate) : nullptr;
    a.wmad = p->width_sigma ? (int64_t*)(ws + L.wmad) : nullptr;
    a.sigw = p->width_sigma ? (double*)(ws + L.sigw) : nullptr;
    if (p->width_sigma) {
        p->last_sigw = a.sigw;
        p->last_wmad = a.wmad;
    }
    return a;
}

RfiArgs make_rfi_args(hp_plan* p, const Layout& L, uint8_t* ws, const uint8_t* x, uint8_t* xt,
                      int64_t xt_pitch, int64_t nsamps, uint8_t* out) {
    RfiArgs r;
    r.x = x;
    r.xt = xt;
    r.xt_pitch = xt_pitch;
    r.nsamps = nsamps;
    r.nch = p->nchans;
    r.nb_k = p->rfi_nb_k;
    r.hist = (uint32_t*)(ws + L.r_hist);
    r.med = (int32_t*)(ws + L.r_med);
    r.spread = (int32_t*)(ws + L.r_spread);
    r.chan_flag = ws + L.r_cflag;
    r.samp_flag = ws + L.r_sflag;
    r.one = (int32_t*)(ws + L.r_one);
    r.out = out;
    // the zero-DM series as a one-trial, one-width (W = 1) stats-only search
    SearchArgs& z = r.z;
    std::memset(&z, 0, sizeof(z));
    int32_t* zs = (int32_t*)(ws + L.r_z);
    z.D = zs;
    z.pitch = L.r_zpitch;
    z.nout = nsamps;
    z.ndm = 1;
    z.nw = 1;
    z.widths = r.one;
    z.wmax = 1;
    z.thr = p->rfi_bb_k;
    z.baseline_mode = p->baseline_mode;
    z.win = baseline_window(p);
    z.levels = remedian_levels(z.win);
    z.lvl_a = (int32_t*)(ws + L.r_lvl_a);
    z.lvl_b = (int32_t*)(ws + L.r_lvl_b);
    z.lvl_pitch_a = L.r_lvl_pitch_a;
    z.lvl_pitch_b = L.r_lvl_pitch_b;
    z.mean_pre = (int64_t*)(ws + L.r_mean);
    z.mean_pitch = L.r_mean_pitch;
    z.hist = (uint32_t*)(ws + L.r_zhist);
    z.refine_bucket = (int32_t*)(ws + L.r_bucket);
    z.refine_rank = (int64_t*)(ws + L.r_rank);
    z.mad = (int64_t*)(ws + L.r_mad);
    z.sigma = (double*)(ws + L.r_sigma);
    z.tint = (int64_t*)(ws + L.r_tint);
    z.status = p->status;
    z.Y = p->baseline_mode == 1 ? (int32_t*)(ws + L.r_y) : zs;   // in place in median mode
    z.ypitch = L.r_zpitch;
    z.nwin = nsamps;
    z.stats_only = 1;
    z.sample_mul = 1;
    return r;
}

MergeArgs make_merge_args(hp_plan* p, const Layout& L, uint8_t* ws, const hp_raw_cand* raw,
                          const int64_t* nraw, int64_t cap, const double* sigma,
                          hp_cand_buf* out) {
    MergeArgs m;
    m.raw = raw;
    m.nraw = nraw;
    m.cap = cap;
    m.sigma = sigma;
    m.sigw = nullptr;   // set by the callers that searched with per-width sigmas
    m.widths = p->d_widths;
    m.nw = p->nw();
    m.wmax = p->wmax;
    m.dm_tol = p->dm_tol;
    m.t_gap = p->t_gap;
    m.w_tol = p->w_tol;
    m.keys[0] = (uint64_t*)(ws + L.keys0);
    m.keys[1] = (uint64_t*)(ws + L.keys1);
    m.vals[0] = (int64_t*)(ws + L.vals0);
    m.vals[1] = (int64_t*)(ws + L.vals1);
    m.parent = (int32_t*)(ws + L.parent);
    m.best_bits = (uint64_t*)(ws + L.best);
    m.rep = (int32_t*)(ws + L.rep);
    m.members = (int32_t*)(ws + L.members);
    m.dm_lo = (int32_t*)(ws + L.dmlo);
    m.dm_hi = (int32_t*)(ws + L.dmhi);
    m.t_lo = (unsigned long long*)(ws + L.tlo);
    m.t_hi = (unsigned long long*)(ws + L.thi);
    m.scan = (int32_t*)(ws + L.scan);
    m.block_sums = (int32_t*)(ws + L.bsums);
    m.n_clamped = (int64_t*)(ws + L.nclamp);
    m.trial_start = (int64_t*)(ws + L.tstart);
    m.ndm = p->ndm();
    m.out = out->data;
    m.out_cap = out->capacity;
    m.out_count = out->count;
    m.status = p->status;
    return m;
}

// The autotuner's search space: the byte-row kernels (every earlier layout is
// slower on every shape measured and stays selectable by hand).
bool autotune_candidate(int c) { return c >= 0 && c < kNumDedispConfigs; }

// time one transpose + dedispersion of `p` on `s` with events (synchronising)
int time_dedisp(hp_plan* p, const uint8_t* fb, int64_t nsamps, cudaStream_t s, int reps,
                float* ms_out) {
    int rc = ensure_device_tables(p, s);
    if (rc) return rc;
    Layout L = make_layout(p, nsamps, true);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return HP_ERR_CUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return HP_ERR_CUDA; }
    const bool timing = p->timing;
    p->timing = false;
    rc = run_dedisp(p, fb, nsamps, L, ws, (int32_t*)(ws + L.D), L.dpitch, s, false, false);
    if (!rc) rc = check_cuda(cudaEventRecord(e0, s));
    for (int r = 0; r < reps && !rc; ++r)
        rc = run_dedisp(p, fb, nsamps, L, ws, (int32_t*)(ws + L.D), L.dpitch, s, false, false);
    if (!rc) rc = check_cuda(cudaEventRecord(e1, s));
    if (!rc) rc = check_cuda(cudaEventSynchronize(e1));
    float ms = 0.f;
    if (!rc) rc = check_cuda(cudaEventElapsedTime(&ms, e0, e1));
    p->timing = timing;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    *ms_out = ms / (float)reps;
    return rc;
}

}  // namespace

// ================================================================ batching
struct hp_batch {
    std::vector<hp_plan*> plans;
    int cfg = hp::kDefaultDedispConfig;
    std::vector<cudaStream_t> side;
    std::vector<cudaEvent_t> done;
    std::vector<cudaEvent_t> dd_done;  // file i dedispersed (its search may start)
    cudaEvent_t fork = nullptr;
    // graph of the last argument set
    cudaGraphExec_t exec = nullptr;
    std::vector<uintptr_t> key;
    int seen = 0;                     // calls made with `key`
    int64_t kernels = 0;              // kernels enqueued per call
};

namespace {

void batch_drop_graph(hp_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    b->key.clear();
    b->seen = 0;
}

int batch_prepare(hp_batch* b, const uint8_t* const* fbs, const int64_t* nsamps, cudaStream_t s,
                  std::vector<Layout>* layouts, std::vector<uint8_t*>* wss) {
    const int n = (int)b->plans.size();
    layouts->resize(n);
    wss->resize(n);
    for (int i = 0; i < n; ++i) {
        hp_plan* p = b->plans[i];
        int rc = validate_search_input(p, fbs ? fbs[i] : nullptr, nsamps[i]);
        if (rc) return rc;
        if (p->sb_chans <= 0) p->dedisp_cfg = b->cfg;   // sub-band files keep their stage-1 shape
        rc = ensure_device_tables(p, s);
        if (rc) return rc;
        (*layouts)[i] = make_layout(p, nsamps[i], true);
        rc = prepare_patterns(p, (*layouts)[i].nout, 1, s);
        if (rc) return rc;
        rc = ensure_workspace(p, (*layouts)[i].total, &(*wss)[i]);
        if (rc) return rc;
    }
    return HP_OK;
}

// The direct dedispersion of one file of a batch.
int batch_dedisp(hp_batch* b, int i, const Layout& L, uint8_t* ws, bool fuse, cudaStream_t s) {
    hp_plan* p = b->plans[i];
    DedispBatch db;
    std::memset(&db, 0, sizeof(db));
    db.njobs = 1;
    db.jobs[0] = make_job(p, ws + L.xt, L.xt_pitch, (int32_t*)(ws + L.D), L.dpitch, L.nout,
                          use_patterns(p, &L.nout, &L.xt_pitch, 1));
    if (fuse) fuse_levels(db.jobs[0], L, ws);
    db.prefix[1] = (int64_t)db.jobs[0].ntt * db.jobs[0].ndt;
    int rc = split_tail(p, &db, s);
    if (!rc) rc = check_cuda(launch_dedisp(b->cfg, db, p->status, p->timeout_ns, s));
    if (!rc) p->last_kernel = launched_kernel(db);
    return rc;
}

// One call of a batch: one transpose launch over every file; then the files'
// dedispersion launches one after another on the caller's stream, largest
// first, and each file's search and merge on its own side stream as soon as
// its dedispersion is done -- so every search runs beside the dedispersion of
// the files after it (the search stage is bound by HBM bandwidth, the
// dedispersion by the integer and shared-memory pipes) -- joined back at the end.
int batch_enqueue(hp_batch* b, const uint8_t* const* fbs, const int64_t* nsamps, cudaStream_t s,
                  hp_cand_buf* outs, const std::vector<Layout>& Ls,
                  const std::vector<uint8_t*>& wss, int64_t* kernels) {
    const int n = (int)b->plans.size();
    TransposeBatch tb;
    std::memset(&tb, 0, sizeof(tb));
    tb.njobs = n;
    std::vector<int> order;
    std::vector<int64_t> work(n, 0);
    for (int i = 0; i < n; ++i) {
        hp_plan* p = b->plans[i];
        const Layout& L = Ls[i];
        tb.jobs[i] = make_transpose_job(fbs[i], nsamps[i], p->nchans, wss[i] + L.xt, L.xt_pitch);
        tb.prefix[i + 1] = tb.prefix[i] + tb.jobs[i].ttiles * tb.jobs[i].ctiles;
        if (p->sb_chans <= 0 && !reach_ok(p, L.nout, L.xt_pitch)) return HP_ERR_INVALID_ARG;
        work[i] = (int64_t)p->ndm() * p->nchans * std::max<int64_t>(L.nout, 0);
        order.push_back(i);
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return work[x] > work[y]; });
    int64_t k = 0;
    int rc = check_cuda(launch_transpose_batch(tb, s));
    if (rc) return rc;
    ++k;
    for (int i = 0; i < n; ++i) {          // RFI mitigation of the files that ask for it
        hp_plan* p = b->plans[i];
        if (!p->rfi) continue;
        const Layout& L = Ls[i];
        const RfiArgs r = make_rfi_args(p, L, wss[i], fbs[i], wss[i] + L.xt, L.xt_pitch,
                                        nsamps[i], nullptr);
        rc = check_cuda(launch_rfi(r, s, &k));
        if (rc) return rc;
    }
    for (int i : order) {
        hp_plan* p = b->plans[i];
        const Layout& L = Ls[i];
        uint8_t* ws = wss[i];
        if (p->sb_chans > 0) {             // the sub-band variant runs its own two stages
            const int64_t before = p->launches;
            rc = run_subband(p, L, ws, (int32_t*)(ws + L.D), L.dpitch, s);
            if (rc) return rc;
            k += p->launches - before;
        } else {
            rc = batch_dedisp(b, i, L, ws, true, s);
            if (rc) return rc;
            ++k;
        }
        rc = check_cuda(cudaEventRecord(b->dd_done[i], s));
        if (rc) return rc;
        cudaStream_t si = b->side[i];
        rc = check_cuda(cudaStreamWaitEvent(si, b->dd_done[i], 0));
        if (rc) return rc;
        hp_raw_cand* raw = (hp_raw_cand*)(ws + L.raw);
        int64_t* raw_count = (int64_t*)(ws + L.raw_count);
        SearchArgs a = make_search_args(p, L, ws, (int32_t*)(ws + L.D), L.dpitch, L.nout, raw,
                                        p->raw_capacity, raw_count);
        if (p->sb_chans <= 0) fuse_levels(a, L, ws, b->cfg);
        rc = check_cuda(launch_search(a, si, &k));
        if (rc) return rc;
        MergeArgs m = make_merge_args(p, L, ws, raw, raw_count, p->raw_capacity, a.sigma, &outs[i]);
        m.sigw = a.width_sigma ? a.sigw : nullptr;
        rc = check_cuda(launch_merge(m, si, &k));
        if (rc) return rc;
        rc = check_cuda(cudaEventRecord(b->done[i], si));
        if (rc) return rc;
    }
    for (int i = 0; i < n; ++i) {
        rc = check_cuda(cudaStreamWaitEvent(s, b->done[i], 0));
        if (rc) return rc;
    }
    *kernels = k;
    return HP_OK;
}

std::vector<uintptr_t> batch_key(const hp_batch* b, const uint8_t* const* fbs,
                                 const int64_t* nsamps, cudaStream_t s, const hp_cand_buf* outs,
                                 const std::vector<uint8_t*>& wss) {
    std::vector<uintptr_t> k;
    k.push_back((uintptr_t)s);
    k.push_back((uintptr_t)b->cfg);
    for (size_t i = 0; i < b->plans.size(); ++i) {
        const hp_plan* p = b->plans[i];
        k.push_back((uintptr_t)fbs[i]);
        k.push_back((uintptr_t)nsamps[i]);
        k.push_back((uintptr_t)outs[i].data);
        k.push_back((uintptr_t)outs[i].capacity);
        k.push_back((uintptr_t)outs[i].count);
        k.push_back((uintptr_t)wss[i]);
        k.push_back((uintptr_t)p->tables);
        k.push_back((uintptr_t)p->ptables);
        k.push_back((uintptr_t)p->baseline_mode);
        k.push_back((uintptr_t)(p->baseline_s * 1e9));
        k.push_back((uintptr_t)p->dm_tol);
        k.push_back((uintptr_t)p->t_gap);
        k.push_back((uintptr_t)p->w_tol);
        k.push_back((uintptr_t)p->raw_capacity);
        k.push_back((uintptr_t)p->timeout_ns);
        k.push_back((uintptr_t)p->rfi);
        k.push_back((uintptr_t)p->rfi_nb_k);
        k.push_back((uintptr_t)(p->rfi_bb_k * 1e6));
        k.push_back((uintptr_t)p->width_sigma);
        k.push_back((uintptr_t)p->sb_chans);
        k.push_back((uintptr_t)p->decimate);
        k.push_back((uintptr_t)p->sb_group);
        k.push_back((uintptr_t)p->fuse_levels);
    }
    return k;
}

}  // namespace

// ====================================================================== ABI
extern "C" {

const char* hp_status_str(int status) {
    switch (status) {
        case HP_OK: return "HP_OK";
        case HP_ERR_INVALID_ARG: return "HP_ERR_INVALID_ARG";
        case HP_ERR_CUDA: return "HP_ERR_CUDA";
        case HP_ERR_OOM: return "HP_ERR_OOM";
        case HP_ERR_CAND_OVERFLOW: return "HP_ERR_CAND_OVERFLOW";
        case HP_ERR_TIMEOUT: return "HP_ERR_TIMEOUT";
        case HP_ERR_NSAMPS_TOO_SHORT: return "HP_ERR_NSAMPS_TOO_SHORT";
        default: return "HP_ERR_UNKNOWN";
    }
}

int hp_plan_create(hp_plan** out, int nchans, double f_top_MHz, double chan_bw_MHz,
                   double tsamp_s, const float* dm_list, int ndm, const int* boxcar_widths,
                   int nw, float snr_threshold) {
    if (!out) return HP_ERR_INVALID_ARG;
    *out = nullptr;
    if (nchans < 1 || nchans > kMaxChans) return HP_ERR_INVALID_ARG;
    if (!std::isfinite(f_top_MHz) || !(f_top_MHz > 0.0)) return HP_ERR_INVALID_ARG;
    if (!std::isfinite(chan_bw_MHz) || !(chan_bw_MHz < 0.0)) return HP_ERR_INVALID_ARG;
    if (!(f_top_MHz + (double)(nchans - 1) * chan_bw_MHz > 0.0)) return HP_ERR_INVALID_ARG;
    if (!std::isfinite(tsamp_s) || !(tsamp_s > 0.0)) return HP_ERR_INVALID_ARG;
    if (!dm_list || ndm < 1 || ndm > kMaxDMs) return HP_ERR_INVALID_ARG;
    if (!boxcar_widths || nw < 1 || nw > kMaxWidths) return HP_ERR_INVALID_ARG;
    if (!std::isfinite(snr_threshold) || !(snr_threshold > 0.0f)) return HP_ERR_INVALID_ARG;
    for (int d = 0; d < ndm; ++d) {
        if (!std::isfinite(dm_list[d]) || dm_list[d] < 0.0f) return HP_ERR_INVALID_ARG;
        if (d > 0 && dm_list[d] < dm_list[d - 1]) return HP_ERR_INVALID_ARG;
    }
    for (int k = 0; k < nw; ++k) {
        if (boxcar_widths[k] < 1 || boxcar_widths[k] > kMaxWidth) return HP_ERR_INVALID_ARG;
        if (k > 0 && boxcar_widths[k] <= boxcar_widths[k - 1]) return HP_ERR_INVALID_ARG;
    }
    hp_plan* p = new (std::nothrow) hp_plan;
    if (!p) return HP_ERR_OOM;
    p->nchans = nchans;
    p->f_top = f_top_MHz;
    p->chan_bw = chan_bw_MHz;
    p->tsamp = tsamp_s;
    p->dm_list.assign(dm_list, dm_list + ndm);
    p->widths.assign(boxcar_widths, boxcar_widths + nw);
    p->thr = snr_threshold;
    p->w_tol = nw;
    p->wmax = boxcar_widths[nw - 1];
    compute_delays(p);
    // the sum of nchans bytes must fit int32 and every delay must be reachable
    if ((int64_t)nchans * 255 > INT32_MAX || p->maxd >= kMaxSamples) {
        delete p;
        return HP_ERR_INVALID_ARG;
    }
    *out = p;
    return HP_OK;
}

int hp_plan_destroy(hp_plan* p) {
    if (!p) return HP_OK;
    bool any_ev = false;
    for (int st = 0; st < HP_NUM_STAGES; ++st) any_ev = any_ev || !p->ev[st].empty();
    if (p->tables || p->ptables || p->ws_own || any_ev) cudaDeviceSynchronize();
    plan_free(p, p->tables, p->tables_bytes);
    plan_free(p, p->ptables, p->ptables_bytes);
    plan_free(p, p->ws_own, p->ws_own_bytes);
    for (int st = 0; st < HP_NUM_STAGES; ++st)
        for (cudaEvent_t e : p->ev[st]) cudaEventDestroy(e);
    delete p;
    return HP_OK;
}

int hp_plan_set_param(hp_plan* p, int param, double v) {
    if (!p || !std::isfinite(v)) return HP_ERR_INVALID_ARG;
    switch (param) {
        case HP_PARAM_BASELINE_MODE:
            if (v != 0.0 && v != 1.0) return HP_ERR_INVALID_ARG;
            p->baseline_mode = (int)v;
            return HP_OK;
        case HP_PARAM_BASELINE_S:
            if (!(v > 0.0)) return HP_ERR_INVALID_ARG;
            p->baseline_s = v;
            return HP_OK;
        case HP_PARAM_DM_TOL:
            if (v < 0 || v > kMaxDMs || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->dm_tol = (int)v;
            return HP_OK;
        case HP_PARAM_T_GAP:
            if (std::fabs(v) > (double)kMaxMergeGap || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->t_gap = (int64_t)v;
            return HP_OK;
        case HP_PARAM_W_TOL:
            if (v < 0 || v > kMaxWidths || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->w_tol = (int)v;
            return HP_OK;
        case HP_PARAM_RAW_CAPACITY:
            if (v < 1024 || v > (double)((int64_t)1 << 30) || v != std::floor(v))
                return HP_ERR_INVALID_ARG;
            p->raw_capacity = (int64_t)v;
            return HP_OK;
        case HP_PARAM_DEDISP_CONFIG:
            if (v < 0 || v >= kNumDedispConfigs || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->dedisp_cfg = (int)v;
            p->dedisp_cfg_set = true;
            return HP_OK;
        case HP_PARAM_STAGE_TIMING:
            if (v != 0.0 && v != 1.0) return HP_ERR_INVALID_ARG;
            p->timing = v != 0.0;
            return HP_OK;
        case HP_PARAM_TIMEOUT_S:
            if (!(v > 0.0) || v > 3600.0) return HP_ERR_INVALID_ARG;
            p->timeout_ns = (uint64_t)(v * 1e9);
            return HP_OK;
        case HP_PARAM_RFI:
            if (v != 0.0 && v != 1.0) return HP_ERR_INVALID_ARG;
            p->rfi = v != 0.0;
            return HP_OK;
        case HP_PARAM_RFI_NB_K:
            if (v < 0 || v > 255 || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->rfi_nb_k = (int)v;
            return HP_OK;
        case HP_PARAM_RFI_BB_K:
            if (!(v > 0.0) || v > 1e6) return HP_ERR_INVALID_ARG;
            p->rfi_bb_k = (float)v;
            return HP_OK;
        case HP_PARAM_DECIMATE:
            // a block size q = W / R of at most 1024 keeps the summed series int32
            if (v < 0 || v != std::floor(v) || (v > 0 && p->wmax / v > 1024)) return HP_ERR_INVALID_ARG;
            p->decimate = (int)v;
            return HP_OK;
        case HP_PARAM_WIDTH_SIGMA:
            if (v != 0.0 && v != 1.0) return HP_ERR_INVALID_ARG;
            p->width_sigma = v == 1.0;
            p->last_sigw = nullptr;
            p->last_wmad = nullptr;
            return HP_OK;
        case HP_PARAM_SUBBAND_CHANS:
            if (v < 0 || v > p->nchans || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->sb_chans = (int)v;
            if (!p->dedisp_cfg_set)
                p->dedisp_cfg = p->sb_chans > 0 ? kDefaultSubbandConfig : kDefaultDedispConfig;
            apply_subband(p);
            return HP_OK;
        case HP_PARAM_FUSE_LEVELS:
            if (v != 0.0 && v != 1.0) return HP_ERR_INVALID_ARG;
            p->fuse_levels = v == 1.0;
            return HP_OK;
        case HP_PARAM_SUBBAND_GROUP:
            if (v < 1 || v > p->ndm() || v != std::floor(v)) return HP_ERR_INVALID_ARG;
            p->sb_group = (int)v;
            apply_subband(p);
            return HP_OK;
        default:
            return HP_ERR_INVALID_ARG;
    }
}

int hp_plan_get_param(const hp_plan* p, int param, double* v) {
    if (!p || !v) return HP_ERR_INVALID_ARG;
    switch (param) {
        case HP_PARAM_BASELINE_MODE: *v = p->baseline_mode; return HP_OK;
        case HP_PARAM_BASELINE_S: *v = p->baseline_s; return HP_OK;
        case HP_PARAM_DM_TOL: *v = p->dm_tol; return HP_OK;
        case HP_PARAM_T_GAP: *v = (double)p->t_gap; return HP_OK;
        case HP_PARAM_W_TOL: *v = p->w_tol; return HP_OK;
        case HP_PARAM_RAW_CAPACITY: *v = (double)p->raw_capacity; return HP_OK;
        case HP_PARAM_DEDISP_CONFIG: *v = p->dedisp_cfg; return HP_OK;
        case HP_PARAM_STAGE_TIMING: *v = p->timing ? 1.0 : 0.0; return HP_OK;
        case HP_PARAM_TIMEOUT_S: *v = (double)p->timeout_ns * 1e-9; return HP_OK;
        case HP_PARAM_RFI: *v = p->rfi ? 1.0 : 0.0; return HP_OK;
        case HP_PARAM_RFI_NB_K: *v = p->rfi_nb_k; return HP_OK;
        case HP_PARAM_RFI_BB_K: *v = (double)p->rfi_bb_k; return HP_OK;
        case HP_PARAM_SUBBAND_CHANS: *v = p->sb_chans; return HP_OK;
        case HP_PARAM_WIDTH_SIGMA: *v = p->width_sigma ? 1.0 : 0.0; return HP_OK;
        case HP_PARAM_DECIMATE: *v = p->decimate; return HP_OK;
        case HP_PARAM_SUBBAND_GROUP: *v = p->sb_group; return HP_OK;
        case HP_PARAM_FUSE_LEVELS: *v = p->fuse_levels ? 1.0 : 0.0; return HP_OK;
        default: return HP_ERR_INVALID_ARG;
    }
}

int hp_plan_delays(const hp_plan* p, int32_t* out_host) {
    if (!p || !out_host) return HP_ERR_INVALID_ARG;
    const std::vector<int32_t>& t = p->sb_chans > 0 ? p->sb_eff : p->delays;
    std::memcpy(out_host, t.data(), t.size() * sizeof(int32_t));
    return HP_OK;
}

int hp_plan_max_delay(const hp_plan* p, int32_t* max_delay) {
    if (!p || !max_delay) return HP_ERR_INVALID_ARG;
    *max_delay = p->maxd;
    return HP_OK;
}

int hp_plan_workspace_bytes(const hp_plan* p, int64_t nsamps, size_t* bytes) {
    if (!p || !bytes) return HP_ERR_INVALID_ARG;
    if (nsamps <= (int64_t)p->maxd + p->wmax) return HP_ERR_NSAMPS_TOO_SHORT;
    *bytes = make_layout(p, nsamps, true).total;
    return HP_OK;
}

int hp_plan_set_allocator(hp_plan* p, hp_alloc_fn alloc, hp_free_fn free_fn, void* ctx) {
    if (!p || (alloc == nullptr) != (free_fn == nullptr)) return HP_ERR_INVALID_ARG;
    if (p->tables || p->ptables || p->ws_own) {
        // return what the previous allocator gave (the tables keep the status word)
        int st = 0;
        if (p->status) cudaMemcpy(&st, p->status, sizeof(int), cudaMemcpyDeviceToHost);
        cudaDeviceSynchronize();
        plan_free(p, p->tables, p->tables_bytes);
        plan_free(p, p->ptables, p->ptables_bytes);
        plan_free(p, p->ws_own, p->ws_own_bytes);
        p->ptables = nullptr;
        p->ptables_bytes = 0;
        p->ptiling = DedispTiling();   // built again on the next use
        p->tables = nullptr;
        p->tables_bytes = 0;
        p->tables_cfg = -1;
        p->status = nullptr;
        p->ws_own = nullptr;
        p->ws_own_bytes = 0;
        if (st != 0) p->pending_status = st;
    }
    if (!p->ptables) p->pat_estimate = PatternCost();   // the new allocator may have room for the tables
    p->alloc_fn = alloc;
    p->free_fn = free_fn;
    p->alloc_ctx = ctx;
    return HP_OK;
}

int hp_plan_bind_workspace(hp_plan* p, void* ws, size_t bytes) {
    if (!p) return HP_ERR_INVALID_ARG;
    if (ws && ((uintptr_t)ws & 255u)) return HP_ERR_INVALID_ARG;
    p->ws_user = ws;
    p->ws_user_bytes = ws ? bytes : 0;
    return HP_OK;
}

int hp_plan_prepare(hp_plan* p, int64_t nsamps, void* stream) {
    int rc = validate_search_input(p, p, nsamps);   // (the plan stands for the input's pointer)
    if (rc) return rc;
    rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    const Layout L = make_layout(p, nsamps, true);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    return prepare_patterns(p, L.nout, 1, (cudaStream_t)stream);
}

int hp_rfi_clean(hp_plan* p, const uint8_t* fb, int64_t nsamps, void* stream, uint8_t* cleaned,
                 uint8_t* chan_flag, uint8_t* samp_flag, int32_t* chan_median) {
    if (!p || !fb || nsamps < 1 || nsamps >= kMaxSamples) return HP_ERR_INVALID_ARG;
    if (cleaned == fb) return HP_ERR_INVALID_ARG;
    int rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    Layout L = make_layout(p, std::max<int64_t>(nsamps, (int64_t)p->maxd + 1), true);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    rc = check_cuda(launch_transpose(fb, nsamps, p->nchans, ws + L.xt, L.xt_pitch, s));
    if (rc) return rc;
    ++p->launches;
    const RfiArgs r = make_rfi_args(p, L, ws, fb, ws + L.xt, L.xt_pitch, nsamps, cleaned);
    rc = check_cuda(launch_rfi(r, s, &p->launches));
    if (rc) return rc;
    if (chan_flag)
        rc = check_cuda(cudaMemcpyAsync(chan_flag, r.chan_flag, (size_t)p->nchans,
                                        cudaMemcpyDeviceToDevice, s));
    if (!rc && samp_flag)
        rc = check_cuda(cudaMemcpyAsync(samp_flag, r.samp_flag, (size_t)nsamps,
                                        cudaMemcpyDeviceToDevice, s));
    if (!rc && chan_median)
        rc = check_cuda(cudaMemcpyAsync(chan_median, r.med, (size_t)p->nchans * 4,
                                        cudaMemcpyDeviceToDevice, s));
    return rc;
}

int hp_dedisperse(hp_plan* p, const uint8_t* fb, int64_t nsamps, int32_t* out, int64_t pitch,
                  void* stream) {
    int rc = validate_search_input(p, fb, nsamps);
    if (rc) return rc;
    const int64_t nout = nsamps - p->maxd;
    if (!out || pitch < nout || (pitch & 3) || ((uintptr_t)out & 15u)) return HP_ERR_INVALID_ARG;
    rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    Layout L = make_layout(p, nsamps, true);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    return run_dedisp(p, fb, nsamps, L, ws, out, pitch, (cudaStream_t)stream, true, false);
}

int hp_detect(hp_plan* p, const int32_t* series, int64_t nout, int64_t pitch, void* stream,
              hp_raw_buf* raw_out, double* sigma_dev, int64_t* mad_dev) {
    if (!p || !series || !raw_out || !raw_out->data || !raw_out->count || raw_out->capacity < 0)
        return HP_ERR_INVALID_ARG;
    if (nout <= p->wmax || pitch < nout) return HP_ERR_NSAMPS_TOO_SHORT;
    int rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    Layout L = make_layout(p, nout + p->maxd, false);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    SearchArgs a = make_search_args(p, L, ws, series, pitch, nout, raw_out->data,
                                    raw_out->capacity, raw_out->count);
    const int ti = stage_begin(p, HP_STAGE_SEARCH, s);
    rc = check_cuda(launch_search(a, s, &p->launches));
    stage_end(p, HP_STAGE_SEARCH, ti, s);
    if (rc) return rc;
    if (sigma_dev)
        rc = check_cuda(cudaMemcpyAsync(sigma_dev, a.sigma, sizeof(double) * p->ndm(),
                                        cudaMemcpyDeviceToDevice, s));
    if (!rc && mad_dev)
        rc = check_cuda(cudaMemcpyAsync(mad_dev, a.mad, sizeof(int64_t) * p->ndm(),
                                        cudaMemcpyDeviceToDevice, s));
    return rc;
}

int hp_merge(hp_plan* p, const hp_raw_cand* raw, const int64_t* nraw, int64_t raw_capacity,
             const double* sigma, void* stream, hp_cand_buf* out) {
    if (!p || !raw || !nraw || !sigma || !out || !out->data || !out->count || out->capacity < 0 ||
        raw_capacity < 0)
        return HP_ERR_INVALID_ARG;
    int rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    // the merge scratch is sized by the plan's raw capacity
    if (raw_capacity > p->raw_capacity) return HP_ERR_INVALID_ARG;
    Layout L = make_layout(p, (int64_t)p->maxd + p->wmax + 1, false);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    MergeArgs m = make_merge_args(p, L, ws, raw, nraw, raw_capacity, sigma, out);
    cudaStream_t s = (cudaStream_t)stream;
    const int ti = stage_begin(p, HP_STAGE_MERGE, s);
    rc = check_cuda(launch_merge(m, s, &p->launches));
    stage_end(p, HP_STAGE_MERGE, ti, s);
    return rc;
}

int hp_search(hp_plan* p, const uint8_t* fb, int64_t nsamps, void* stream, hp_cand_buf* out) {
    int rc = validate_search_input(p, fb, nsamps);
    if (rc) return rc;
    if (!out || !out->data || !out->count || out->capacity < 0) return HP_ERR_INVALID_ARG;
    rc = ensure_device_tables(p, (cudaStream_t)stream);
    if (rc) return rc;
    Layout L = make_layout(p, nsamps, true);
    uint8_t* ws = nullptr;
    rc = ensure_workspace(p, L.total, &ws);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    int32_t* D = (int32_t*)(ws + L.D);
    rc = run_dedisp(p, fb, nsamps, L, ws, D, L.dpitch, s, true, true);
    if (rc) return rc;
    hp_raw_cand* raw = (hp_raw_cand*)(ws + L.raw);
    int64_t* raw_count = (int64_t*)(ws + L.raw_count);
    SearchArgs a = make_search_args(p, L, ws, D, L.dpitch, L.nout, raw, p->raw_capacity, raw_count);
    fuse_levels(a, L, ws, p->dedisp_cfg);
    int ti = stage_begin(p, HP_STAGE_SEARCH, s);
    rc = check_cuda(launch_search(a, s, &p->launches));
    stage_end(p, HP_STAGE_SEARCH, ti, s);
    if (rc) return rc;
    MergeArgs m = make_merge_args(p, L, ws, raw, raw_count, p->raw_capacity, a.sigma, out);
    m.sigw = a.width_sigma ? a.sigw : nullptr;
    ti = stage_begin(p, HP_STAGE_MERGE, s);
    rc = check_cuda(launch_merge(m, s, &p->launches));
    stage_end(p, HP_STAGE_MERGE, ti, s);
    return rc;
}

int hp_width_sigmas(hp_plan* p, double* sigma_w_dev, int64_t* mad_w_dev, void* stream) {
    if (!p || (!sigma_w_dev && !mad_w_dev)) return HP_ERR_INVALID_ARG;
    if (!p->width_sigma || !p->last_sigw) return HP_ERR_INVALID_ARG;
    const size_t pairs = (size_t)p->ndm() * p->nw();
    cudaStream_t s = (cudaStream_t)stream;
    int rc = HP_OK;
    if (sigma_w_dev)
        rc = check_cuda(cudaMemcpyAsync(sigma_w_dev, p->last_sigw, pairs * sizeof(double),
                                        cudaMemcpyDeviceToDevice, s));
    if (!rc && mad_w_dev)
        rc = check_cuda(cudaMemcpyAsync(mad_w_dev, p->last_wmad, pairs * sizeof(int64_t),
                                        cudaMemcpyDeviceToDevice, s));
    return rc;
}

int hp_plan_stats(hp_plan* p, hp_stats* out, int reset) {
    if (!p || !out) return HP_ERR_INVALID_ARG;
    for (int st = 0; st < HP_NUM_STAGES; ++st) {
        double ms = 0.0;
        for (int i = 0; i < p->ev_used[st]; ++i) {
            if (cudaEventSynchronize(p->ev[st][2 * i + 1]) != cudaSuccess) return HP_ERR_CUDA;
            float f = 0.f;
            if (cudaEventElapsedTime(&f, p->ev[st][2 * i], p->ev[st][2 * i + 1]) != cudaSuccess)
                return HP_ERR_CUDA;
            ms += f;
        }
        out->stage_ms[st] = ms;
        out->stage_calls[st] = p->ev_used[st];
        if (reset) p->ev_used[st] = 0;
    }
    out->kernel_launches = p->launches;
    out->device_allocs = p->device_allocs;
    if (reset) p->launches = 0;
    return HP_OK;
}

int hp_plan_dedisp_kernel(const hp_plan* p, int* kernel) {
    if (!p || !kernel || p->last_kernel < 0) return HP_ERR_INVALID_ARG;
    *kernel = p->last_kernel;
    return HP_OK;
}

int hp_plan_autotune(hp_plan* p, const uint8_t* fb, int64_t nsamps, void* stream,
                     int* best_config, float* best_ms) {
    int rc = validate_search_input(p, fb, nsamps);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const int keep = p->dedisp_cfg;
    int best = -1;
    float best_t = 0.f;
    for (int c = 0; c < kNumDedispConfigs; ++c) {
        if (!autotune_candidate(c)) continue;
        p->dedisp_cfg = c;
        float ms = 0.f;
        rc = time_dedisp(p, fb, nsamps, s, 2, &ms);
        if (rc == HP_ERR_INVALID_ARG) continue;     // this tile shape cannot hold the rows
        if (rc) { p->dedisp_cfg = keep; return rc; }
        if (best < 0 || ms < best_t) { best = c; best_t = ms; }
    }
    p->dedisp_cfg = best >= 0 ? best : keep;
    if (best >= 0) p->dedisp_cfg_set = true;
    rc = ensure_device_tables(p, s);
    if (rc) return rc;
    if (best_config) *best_config = p->dedisp_cfg;
    if (best_ms) *best_ms = best_t;
    return best >= 0 ? HP_OK : HP_ERR_INVALID_ARG;
}

int hp_batch_create(hp_batch** out, hp_plan* const* plans, int nfiles) {
    if (!out) return HP_ERR_INVALID_ARG;
    *out = nullptr;
    if (!plans || nfiles < 1 || nfiles > HP_BATCH_MAX_FILES || nfiles > kMaxJobs)
        return HP_ERR_INVALID_ARG;
    for (int i = 0; i < nfiles; ++i)
        if (!plans[i]) return HP_ERR_INVALID_ARG;
    hp_batch* b = new (std::nothrow) hp_batch;
    if (!b) return HP_ERR_OOM;
    b->plans.assign(plans, plans + nfiles);
    // the direct files' tile shape: the first direct file's (sub-band files keep theirs)
    b->cfg = kDefaultDedispConfig;
    for (int i = nfiles - 1; i >= 0; --i)
        if (plans[i]->sb_chans <= 0) b->cfg = plans[i]->dedisp_cfg;
    int rc = HP_OK;
    if (cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming) != cudaSuccess) rc = HP_ERR_CUDA;
    for (int i = 0; i < nfiles && !rc; ++i) {
        cudaStream_t st;
        cudaEvent_t ev;
        if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) { rc = HP_ERR_CUDA; break; }
        b->side.push_back(st);
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) { rc = HP_ERR_CUDA; break; }
        b->done.push_back(ev);
        if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) { rc = HP_ERR_CUDA; break; }
        b->dd_done.push_back(ev);
    }
    if (rc) {
        hp_batch_destroy(b);
        return rc;
    }
    *out = b;
    return HP_OK;
}

int hp_batch_destroy(hp_batch* b) {
    if (!b) return HP_OK;
    cudaDeviceSynchronize();
    batch_drop_graph(b);
    for (cudaStream_t st : b->side) cudaStreamDestroy(st);
    for (cudaEvent_t ev : b->done) cudaEventDestroy(ev);
    for (cudaEvent_t ev : b->dd_done) cudaEventDestroy(ev);
    if (b->fork) cudaEventDestroy(b->fork);
    delete b;
    return HP_OK;
}

int hp_batch_set_config(hp_batch* b, int config) {
    if (!b || config < 0 || config >= kNumDedispConfigs) return HP_ERR_INVALID_ARG;
    if (config != b->cfg) batch_drop_graph(b);
    b->cfg = config;
    return HP_OK;
}

int hp_batch_search(hp_batch* b, const uint8_t* const* fbs, const int64_t* nsamps, void* stream,
                    hp_cand_buf* outs) {
    if (!b || !fbs || !nsamps || !outs) return HP_ERR_INVALID_ARG;
    const int n = (int)b->plans.size();
    for (int i = 0; i < n; ++i)
        if (!outs[i].data || !outs[i].count || outs[i].capacity < 0) return HP_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<Layout> Ls;
    std::vector<uint8_t*> wss;
    int rc = batch_prepare(b, fbs, nsamps, s, &Ls, &wss);
    if (rc) return rc;
    const std::vector<uintptr_t> key = batch_key(b, fbs, nsamps, s, outs, wss);
    if (key != b->key) {
        batch_drop_graph(b);
        b->key = key;
    }
    if (b->exec) return check_cuda(cudaGraphLaunch(b->exec, s));
    if (b->seen++ == 0 || s == nullptr) {
        // first call with these arguments: run directly (kernel attributes are
        // set outside any capture); the legacy default stream cannot be captured
        return batch_enqueue(b, fbs, nsamps, s, outs, Ls, wss, &b->kernels);
    }
    rc = check_cuda(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    if (rc) return rc;
    const int erc = batch_enqueue(b, fbs, nsamps, s, outs, Ls, wss, &b->kernels);
    cudaGraph_t g = nullptr;
    rc = check_cuda(cudaStreamEndCapture(s, &g));
    if (erc) {
        if (g) cudaGraphDestroy(g);
        return erc;
    }
    if (rc) return rc;
    rc = check_cuda(cudaGraphInstantiate(&b->exec, g, 0));
    cudaGraphDestroy(g);
    if (rc) {
        b->exec = nullptr;
        return rc;
    }
    return check_cuda(cudaGraphLaunch(b->exec, s));
}

int hp_batch_autotune(hp_batch* b, const uint8_t* const* fbs, const int64_t* nsamps, void* stream,
                      int* best_config, float* best_ms) {
    if (!b || !fbs || !nsamps) return HP_ERR_INVALID_ARG;
    for (hp_plan* p : b->plans)
        if (p->sb_chans > 0) return HP_ERR_INVALID_ARG;   // direct dedispersion only
    cudaStream_t s = (cudaStream_t)stream;
    const int n = (int)b->plans.size();
    const int keep = b->cfg;
    int best = -1;
    float best_t = 0.f;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return HP_ERR_CUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return HP_ERR_CUDA; }
    int rc = HP_OK;
    bool warm = false;
    for (int c = 0; c < kNumDedispConfigs; ++c) {
        if (!autotune_candidate(c)) continue;
        b->cfg = c;
        std::vector<Layout> Ls;
        std::vector<uint8_t*> wss;
        rc = batch_prepare(b, fbs, nsamps, s, &Ls, &wss);
        if (rc == HP_ERR_INVALID_ARG) { rc = HP_OK; continue; }
        if (rc) break;
        TransposeBatch tb;
        std::memset(&tb, 0, sizeof(tb));
        tb.njobs = n;
        bool reach = true;
        for (int i = 0; i < n; ++i) {
            hp_plan* p = b->plans[i];
            const Layout& L = Ls[i];
            reach = reach && reach_ok(p, L.nout, L.xt_pitch);
            tb.jobs[i] = make_transpose_job(fbs[i], nsamps[i], p->nchans, wss[i] + L.xt, L.xt_pitch);
            tb.prefix[i + 1] = tb.prefix[i] + tb.jobs[i].ttiles * tb.jobs[i].ctiles;
        }
        if (!reach) continue;          // this tile shape cannot stage these rows
        // the launches that a search makes
        auto pass = [&]() {
            int r = check_cuda(launch_transpose_batch(tb, s));
            for (int i = 0; i < n && !r; ++i) r = batch_dedisp(b, i, Ls[i], wss[i], false, s);
            return r;
        };
        if (!warm) {   // one untimed pass before the first timed one
            rc = pass();
            warm = true;
        }
        if (!rc) rc = check_cuda(cudaEventRecord(e0, s));
        if (!rc) rc = pass();
        if (!rc) rc = check_cuda(cudaEventRecord(e1, s));
        if (!rc) rc = check_cuda(cudaEventSynchronize(e1));
        float ms = 0.f;
        if (!rc) rc = check_cuda(cudaEventElapsedTime(&ms, e0, e1));
        if (rc) break;
        if (best < 0 || ms < best_t) { best = c; best_t = ms; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->cfg = best >= 0 ? best : keep;
    batch_drop_graph(b);
    if (rc) return rc;
    for (hp_plan* p : b->plans) {
        if (p->sb_chans <= 0) p->dedisp_cfg = b->cfg;
        rc = ensure_device_tables(p, s);
        if (rc) return rc;
    }
    if (best_config) *best_config = b->cfg;
    if (best_ms) *best_ms = best_t;
    return best >= 0 ? HP_OK : HP_ERR_INVALID_ARG;
}

int hp_batch_sync_status(hp_batch* b, void* stream) {
    if (!b) return HP_ERR_INVALID_ARG;
    int first = HP_OK;
    for (hp_plan* p : b->plans) {
        const int st = hp_plan_sync_status(p, stream);
        if (first == HP_OK && st != HP_OK) first = st;
    }
    return first;
}

int hp_batch_kernels_per_call(const hp_batch* b, int64_t* kernels) {
    if (!b || !kernels) return HP_ERR_INVALID_ARG;
    *kernels = b->kernels;
    return HP_OK;
}

int hp_plan_sync_status(hp_plan* p, void* stream) {
    if (!p) return HP_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaStreamSynchronize(s) != cudaSuccess) return HP_ERR_CUDA;
    if (!p->status) {
        const int st = p->pending_status;
        p->pending_status = 0;
        return st;
    }
    int st = 0;
    if (cudaMemcpy(&st, p->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return HP_ERR_CUDA;
    if (st != 0 && cudaMemset(p->status, 0, sizeof(int)) != cudaSuccess) return HP_ERR_CUDA;
    return st;
}

}  // extern "C"
