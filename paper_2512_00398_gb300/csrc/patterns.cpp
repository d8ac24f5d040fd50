// patterns.cpp -- host tiling of the pattern-row dedispersion kernel
// (patterns.cu): which consecutive channels are summed into shared rows, the
// distinct delay patterns of every DM tile, and the stage tables.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <thread>
#include <vector>

#include "patterns.cuh"
#include "plan_internal.h"

namespace hp {
namespace {

// One distinct pattern of a group: its channels' delays relative to the first
// channel's, and the range of first-channel delays of the trials that use it.
struct Pattern {
    int32_t rel[kPatMaxGroup];
    int32_t lo, hi;
};

struct Group {
    int c = 0, n = 0;               // channels [c, c + n)
    int32_t u0 = 0;                 // sample that chunk 0 starts at (first channel)
    std::vector<Pattern> pats;
    std::vector<int> of_trial;      // pattern of every trial
    int32_t goff[kPatMaxGroup];     // staged window of every channel
    uint32_t nwords[kPatMaxGroup];
};

int chunk_lo(const Pattern& q, int32_t u0) { return (q.lo - u0) / kPatChunk; }
int chunk_hi(const Pattern& q, int32_t u0) {
    return (q.hi - u0 + kPatL + kPatChunk - 1) / kPatChunk;
}

struct TileOut {
    std::vector<StageDesc> stages;
    std::vector<ChanDesc> chans;
    std::vector<uint32_t> tab;
    int64_t max_reach = 0;
    double cost = 0;                // estimated SM cycles per time tile
    bool ok = false;
};

// The tables of one tile.  They are built by a call that waits for them: trying the
// pattern of the trial before first, a channel's delays side by side and one list of
// items a stage instead of vectors in each took the first call of a plan of one tile x
// 1024 channels from 1.82 to 1.22 ms, of 17 tiles from 7.87 to 6.48.
struct TileBuilder {
    const hp_plan* p;
    int d0, nd;
    bool strict;    // bound the tables of a group from above instead of estimating them

    std::vector<int32_t> column;   // delays of the channels from col0 on, nd trials each
    int col0;

    // For channels [begin, end) of trials [d0, d0 + nd).
    TileBuilder(const hp_plan* plan, int first, int n, bool strict_, int begin, int end)
        : p(plan), d0(first), nd(n), strict(strict_), column((size_t)n * (end - begin)), col0(begin) {
        for (int j = 0; j < n; ++j) {
            const int32_t* row = &p->delays[(size_t)(d0 + j) * p->nchans];
            for (int c = begin; c < end; ++c) column[(size_t)(c - begin) * n + j] = row[c];
        }
    }

    // (ascending: the trials are)
    const int32_t* delays(int c) const { return &column[(size_t)(c - col0) * nd]; }
    int32_t delay(int j, int c) const { return delays(c)[j]; }

    // Cost of a group whose sets unpack `sets` chunks in all and put `rows` chunks into
    // rows, by which the channels are cut into groups (about SM cycles: 1620 per group of
    // 15 and 51 chunks at 4096 channels, 24 trials).
    double group_cost(double sets, double rows) const {
        return 150.0 + 21.0 * nd + 21.0 * sets + 13.0 * rows;
    }
    // Its SM cycles, fitted to the 3645 whole-tile launches of plan.cpp (pattern_cycles) that
    // have one wave or tiles alike: measured / estimated 0.97-1.04 (5th to 95th of 100).
    double group_cycles(double sets, double rows) const {
        return 636.0 + 8.7 * nd + 19.5 * sets + 10.6 * rows;
    }

    void make_group(int c, int n, Group* g) const {
        g->c = c;
        g->n = n;
        g->pats.clear();
        g->of_trial.assign(nd, 0);
        size_t i = 0;
        for (int j = 0; j < nd; ++j) {
            Pattern q{};
            for (int k = 0; k < n; ++k) q.rel[k] = delay(j, c + k) - delay(j, c);
            q.lo = q.hi = delay(j, c);
            // (mostly the pattern of the trial before)
            if (j == 0 || std::memcmp(g->pats[i].rel, q.rel, sizeof(q.rel)))
                for (i = 0; i < g->pats.size() && std::memcmp(g->pats[i].rel, q.rel, sizeof(q.rel));) ++i;
            if (i == g->pats.size()) g->pats.push_back(q);
            g->pats[i].hi = q.hi;
            g->of_trial[j] = (int)i;
        }
        g->u0 = delay(0, c) & ~3;
        for (int k = 0; k < n; ++k) {
            const int32_t a = delay(0, c + k), b = delay(nd - 1, c + k);
            g->goff[k] = a & ~15;
            g->nwords[k] = (uint32_t)((b - g->goff[k] + kPatBT + 15) / 16 * 4);
        }
    }

    // Slot of channel k of a group of n (PatItem).
    static int slot(int n, int k) { return n > 2 ? k : 2 * k; }

    // The set that starts at pattern i of the order: the patterns up to the returned
    // index, whose shifts differ by no more than their slots allow (lo: the smallest
    // positions in the channels' windows).
    static size_t set_end(const Group& g, const std::vector<int>& ord, size_t i,
                          int32_t (&lo)[kPatMaxGroup]) {
        static const int limit[4] = {0, kPatShift1, kPatShift2, kPatShift2};
        int32_t hi[kPatMaxGroup];
        size_t e = i;
        for (; e < ord.size(); ++e) {
            int32_t l2[kPatMaxGroup], h2[kPatMaxGroup];
            bool fits = true;
            for (int k = 0; k < g.n; ++k) {
                const int32_t at = g.u0 - g.goff[k] + g.pats[ord[e]].rel[k];
                l2[k] = e == i ? at : std::min(lo[k], at);
                h2[k] = e == i ? at : std::max(hi[k], at);
                fits = fits && h2[k] - l2[k] <= limit[slot(g.n, k)];
            }
            if (!fits) break;
            std::copy(l2, l2 + g.n, lo);
            std::copy(h2, h2 + g.n, hi);
        }
        return e;
    }

    // One item of a set: its form cost (instructions, about) orders the items.
    struct Item {
        PatItem d;
        int row, cost;             // its first row in `Items::rows`
    };
    struct Items {
        std::vector<Item> items;
        std::vector<PatRow> rows;
        size_t bytes() const { return items.size() * sizeof(PatItem) + rows.size() * sizeof(PatRow); }
        void clear() {
            items.clear();
            rows.clear();
        }
        // Append those of another list.
        void append(const Items& more) {
            for (Item it : more.items) {
                it.row += (int)rows.size();
                items.push_back(it);
            }
            rows.insert(rows.end(), more.rows.begin(), more.rows.end());
        }
    };

    // The items of a group whose rows start at byte `row` of the row buffer and
    // whose channels' windows start at chan_off in the raw buffer; org: per pattern
    // the row buffer's byte offset of its word 0.
    void make_items(const Group& g, const std::vector<int>& ord, const uint32_t* chan_off, uint32_t row,
                    Items* out, std::vector<uint32_t>* org) const {
        out->clear();
        org->assign(g.pats.size(), 0);
        struct Row { int kind, lo, n; uint32_t row; };
        Row rows[kPatBD];
        for (size_t i = 0; i < ord.size();) {
            int32_t lo[kPatMaxGroup];
            const size_t e = set_end(g, ord, i, lo);
            PatItem d{};
            d.nchan = (uint8_t)g.n;
            for (int k = 0; k < 4; ++k) d.off[k] = chan_off[0] + (uint32_t)(lo[0] & ~3);   // empty slots
            for (int k = 0; k < g.n; ++k) {
                d.off[slot(g.n, k)] = chan_off[k] + (uint32_t)(lo[k] & ~3);
                d.sel[slot(g.n, k)] = (uint16_t)(0x3210u + 0x1111u * (uint32_t)(lo[k] & 3));
            }
            int first = 1 << 30, last = 0, nrows = 0;
            for (; i < e; ++i) {
                const Pattern& q = g.pats[ord[i]];
                int shift[4] = {};
                for (int k = 0; k < g.n; ++k)
                    shift[slot(g.n, k)] = g.u0 - g.goff[k] + q.rel[k] - lo[k];
                Row r;
                r.kind = 9 * shift[1] + 3 * shift[2] + shift[3];
                r.lo = chunk_lo(q, g.u0);
                r.n = chunk_hi(q, g.u0) - r.lo;
                r.row = row;
                (*org)[ord[i]] = row - (uint32_t)r.lo * kPatChunk * 4;
                row += (uint32_t)r.n * kPatChunk * 4;
                first = std::min(first, r.lo);
                last = std::max(last, r.lo + r.n);
                rows[nrows++] = r;
            }
            // items of kPatItem chunks from the first chunk that any pattern covers
            for (int c0 = first; c0 < last; c0 += kPatItem) {
                Item it;
                it.d = d;
                for (int k = 0; k < 4; ++k) it.d.off[k] += (uint32_t)(c0 * kPatChunk);
                it.cost = 200;
                it.row = (int)out->rows.size();
                for (int k = 0; k < nrows; ++k) {
                    const Row& r = rows[k];
                    uint32_t put = 0;
                    for (int q = 0; q < kPatItem; ++q)
                        if (c0 + q >= r.lo && c0 + q < r.lo + r.n) put |= 1u << q;
                    if (put == 0) continue;
                    // (the item may start before the row; those chunks' stores are masked)
                    out->rows.push_back(
                        PatRow{r.row + (uint32_t)((c0 - r.lo + kPatItem - 1) * kPatChunk * 4),
                               (uint16_t)put, (uint16_t)r.kind});
                    it.cost += 32;
                }
                it.d.nrows = (uint8_t)(out->rows.size() - (size_t)it.row);
                if (it.d.nrows) out->items.push_back(it);
            }
        }
    }

    // The same items in another stage: windows and rows start so many bytes further on.
    static void move_items(uint32_t raw, uint32_t row, Items* out, std::vector<uint32_t>* org) {
        for (Item& it : out->items)
            for (uint32_t& off : it.d.off) off += raw;
        for (PatRow& r : out->rows) r.at += row;
        for (uint32_t& o : *org) o += row;
    }

    // The cheapest cut of the channels [begin, nch) into groups of 1 .. kPatMaxGroup;
    // total: its SM cycles.
    bool cut(int begin, int nch, std::vector<uint8_t>* len, double* total) const {
        std::vector<double> best(nch + 1, 0.0), cycles(nch + 1, 0.0);
        len->assign(nch, 0);
        int cls[kPatBD];
        uint64_t keys[kPatBD];             // the patterns, by refinement: class, relative delay
        int32_t lo[kPatBD], hi[kPatBD];    // their ranges of first-channel delays
        for (int c = nch - 1; c >= begin; --c) {
            best[c] = 1e300;
            std::fill(cls, cls + nd, 0);
            const int32_t* first = delays(c);
            const int32_t u0 = first[0] & ~3;
            uint32_t raw = 0;
            int32_t range[kPatMaxGroup];       // of each channel's shift
            for (int n = 1; n <= kPatMaxGroup && c + n <= nch; ++n) {
                // refine the classes by the n-th channel
                const int32_t* nth = delays(c + n - 1);
                const int32_t a = nth[0], b = nth[nd - 1];
                int32_t r_lo = a - first[0], r_hi = r_lo;
                int nkeys = 0, i = 0;
                for (int j = 0; j < nd; ++j) {
                    const int32_t rel = nth[j] - first[j];
                    r_lo = std::min(r_lo, rel);
                    r_hi = std::max(r_hi, rel);
                    const uint64_t key = (uint64_t)cls[j] << 32 | (uint32_t)rel;
                    if (j == 0 || keys[i] != key)   // (mostly that of the trial before)
                        for (i = 0; i < nkeys && keys[i] != key;) ++i;
                    if (i == nkeys) {
                        keys[nkeys++] = key;
                        lo[i] = first[j];
                    }
                    hi[i] = first[j];
                    cls[j] = i;
                }
                raw += (uint32_t)((b - (a & ~15) + kPatBT + 15) / 16 * 16);
                int chunks = 0, span = 0;
                for (int k = 0; k < nkeys; ++k) {
                    Pattern q{};
                    q.lo = lo[k];
                    q.hi = hi[k];
                    const int e = chunk_hi(q, u0);
                    chunks += e - chunk_lo(q, u0);
                    span = std::max(span, e);
                }
                // about as many sets as the widest range of shifts needs
                range[n - 1] = r_hi - r_lo;
                double sets = 1.0;
                for (int k = 1; k < n; ++k)
                    sets = std::max(sets, (range[k] + 1.0) / (slot(n, k) == 1 ? kPatShift1 + 1 : kPatShift2 + 1));
                // (strict: every pattern in a set of its own)
                const double items = strict ? chunks / kPatItem + 2 * nkeys
                                            : 1.3 * sets * (span / kPatItem + 1);
                const double tab = sizeof(PatHeader) + items * sizeof(PatItem) +
                                   (chunks / kPatItem + 2 * nkeys) * sizeof(PatRow);
                if ((size_t)chunks * kPatChunk * 4 > (size_t)kPatRowBytes ||
                    raw > (uint32_t)(kPatRawBytes - kPatTabBytes) || tab > kPatTabBytes - 16)
                    break;   // more channels only add to each
                const double cost = group_cost(sets * (span + 1), chunks) + best[c + n];
                if (cost < best[c]) {
                    best[c] = cost;
                    cycles[c] = group_cycles(sets * (span + 1), chunks) + cycles[c + n];
                    (*len)[c] = (uint8_t)n;
                }
            }
            if ((*len)[c] == 0) return false;
        }
        *total = cycles[begin];
        return true;
    }

    void build(TileOut* out) const {
        std::vector<uint8_t> len;
        const int nch = p->nchans;
        if (!cut(0, nch, &len, &out->cost)) return;
        // the stage being packed
        Items items;
        std::vector<uint32_t> trials;
        StageDesc sd{};
        uint32_t rows = 0, raw = kPatTabBytes, tab = sizeof(PatHeader);
        int groups = 0, held = 0;
        std::vector<int64_t> load(kPatFormWarps, 0);   // cost given to every forming warp so far
        std::vector<int> order, of;                    // items by cost; the forming warp of each
        size_t last_trials = 0;                        // trial table of the last stage emitted
        auto flush_last = [&]() {
            PatTrials h;
            std::memcpy(&h, &out->tab[last_trials], sizeof(h));
            h.flush = 1;
            std::memcpy(&out->tab[last_trials], &h, sizeof(h));
        };
        auto emit = [&]() {
            if (held + (int)sd.nchan > kStageMaxChans) {   // the stage before flushes
                flush_last();
                held = 0;
            }
            held += (int)sd.nchan;
            // the costliest items first, each to the warp with the least work so far
            const int nitems = (int)items.items.size();
            order.resize(nitems);
            of.resize(nitems);
            for (int i = 0; i < nitems; ++i) order[i] = i;
            std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
                return items.items[x].cost > items.items[y].cost;
            });
            int64_t here[kPatFormWarps] = {};
            for (int i : order) {
                int w = 0;
                for (int v = 1; v < kPatFormWarps; ++v)
                    if (here[v] < here[w] || (here[v] == here[w] && load[v] < load[w])) w = v;
                of[i] = w;
                here[w] += items.items[i].cost;
                load[w] += items.items[i].cost;
            }
            tab = (tab + 15) & ~15u;       // copied in 16-byte pieces
            sd.addr_begin = (uint32_t)out->tab.size();
            sd.addr_bytes = tab;
            sd.addr_off = (uint32_t)(sizeof(PatTrials) + trials.size() * 4);
            sd.tx_bytes += tab + sd.addr_off;
            out->tab.resize(out->tab.size() + (sd.addr_bytes + sd.addr_off) / 4);
            uint8_t* base = reinterpret_cast<uint8_t*>(&out->tab[sd.addr_begin]);
            PatHeader h{};
            uint32_t n = 0, b_off = (uint32_t)(sizeof(h) + nitems * sizeof(PatItem));
            for (int w = 0; w < kPatFormWarps; ++w) {
                h.begin[w] = (uint8_t)n;
                for (int i : order) {
                    if (of[i] != w) continue;
                    Item& it = items.items[i];
                    it.d.row_off = (uint16_t)b_off;
                    std::memcpy(base + sizeof(h) + n * sizeof(PatItem), &it.d, sizeof(PatItem));
                    std::memcpy(base + b_off, &items.rows[it.row], it.d.nrows * sizeof(PatRow));
                    b_off += (uint32_t)(it.d.nrows * sizeof(PatRow));
                    ++n;
                }
            }
            h.begin[kPatFormWarps] = (uint8_t)n;
            std::memcpy(base, &h, sizeof(h));
            PatTrials th{};
            th.ngroups = (uint32_t)groups;
            std::memcpy(base + tab, &th, sizeof(th));
            std::memcpy(base + tab + sizeof(th), trials.data(), trials.size() * 4);
            last_trials = sd.addr_begin + tab / 4;
            out->stages.push_back(sd);
            items.clear();
            trials.clear();
            rows = 0;
            raw = kPatTabBytes;
            tab = sizeof(PatHeader);
            groups = 0;
        };
        Group g;
        std::vector<int> ord;
        Items more;
        std::vector<uint32_t> org;
        for (int c = 0; c < nch; c += len[c]) {
            make_group(c, len[c], &g);
            ord.resize(g.pats.size());
            for (size_t i = 0; i < ord.size(); ++i) ord[i] = (int)i;
            std::sort(ord.begin(), ord.end(), [&](int x, int y) {
                return std::lexicographical_compare(g.pats[x].rel, g.pats[x].rel + g.n, g.pats[y].rel,
                                                    g.pats[y].rel + g.n);
            });
            uint32_t grows = 0, graw = 0;
            for (const Pattern& q : g.pats)
                grows += (uint32_t)(chunk_hi(q, g.u0) - chunk_lo(q, g.u0)) * kPatChunk * 4;
            for (int k = 0; k < g.n; ++k) graw += 4 * g.nwords[k];
            uint32_t chan_off[kPatMaxGroup] = {};
            for (int k = 0; k < g.n; ++k) chan_off[k] = k > 0 ? chan_off[k - 1] + 4 * g.nwords[k - 1] : raw;
            make_items(g, ord, chan_off, rows, &more, &org);
            if (groups > 0 && (groups == kPatStageGroups || rows + grows > (uint32_t)kPatRowBytes ||
                               raw + graw > (uint32_t)kPatRawBytes ||
                               tab + more.bytes() + 15 > (uint32_t)kPatTabBytes ||
                               items.items.size() + more.items.size() > 255)) {
                const uint32_t raw_was = raw, rows_was = rows;
                emit();
                move_items(raw - raw_was, rows - rows_was, &more, &org);   // (modulo 2^32)
                for (int k = 0; k < g.n; ++k) chan_off[k] += raw - raw_was;
            }
            if (more.bytes() + tab + 15 > (uint32_t)kPatTabBytes || more.items.size() > 255) return;
            if (groups == 0) {
                sd = StageDesc{};
                sd.chan_begin = (uint32_t)out->chans.size();
            }
            for (int k = 0; k < g.n; ++k) {
                ChanDesc cd;
                cd.c = (uint32_t)(g.c + k);
                cd.goff = g.goff[k];
                cd.offB = chan_off[k];
                cd.nwords = g.nwords[k];
                out->chans.push_back(cd);
                sd.tx_bytes += 4 * g.nwords[k];
                out->max_reach = std::max<int64_t>(out->max_reach, (int64_t)g.goff[k] + 4 * g.nwords[k]);
            }
            sd.nchan += (uint32_t)g.n;
            trials.resize(trials.size() + kPatSumWarps * kPatPlaces);
            uint32_t* t = &trials[trials.size() - kPatSumWarps * kPatPlaces];
            for (int j = 0; j < kPatBD; ++j) {
                const int jj = j < nd ? j : 0;
                t[j / kPatRD * kPatPlaces + j % kPatRD] =
                    org[g.of_trial[jj]] + 4u * (uint32_t)(delay(jj, g.c) - g.u0);
            }
            tab += (uint32_t)more.bytes();
            items.append(more);
            rows += grows;
            raw += graw;
            ++groups;
        }
        emit();
        flush_last();
        out->ok = true;
    }
};

}  // namespace

bool parallel_for(int n, int threads, const std::function<void(int)>& f) {
    std::atomic<int> next{0};
    std::atomic<bool> failed{false};
    auto work = [&]() {
        try {
            for (int i; !failed && (i = next++) < n;) f(i);
        } catch (...) {
            failed = true;
        }
    };
    const int want = std::min({n, threads, (int)std::max(1u, std::thread::hardware_concurrency())});
    std::vector<std::thread> pool;
    try {
        for (int i = 1; i < want; ++i) pool.emplace_back(work);
    } catch (...) {   // fewer threads than wanted
    }
    work();
    for (std::thread& t : pool) t.join();
    return !failed;
}

// (the launches of plan.cpp, pattern_cycles: measured / estimated 0.99-1.02, 5th to 95th of 100)
double byte_row_cycles(double sums) { return sums / 79.0; }

// First trial of DM tile i.
static int pattern_tile(int ndm, int ntiles, int i) { return (int)((int64_t)ndm * i / ntiles); }

PatternCost estimate_patterns(const hp_plan* p) {
    const int ndm = p->ndm(), ntiles = (ndm + kPatBD - 1) / kPatBD;
    const int nd = std::min(ntiles, 5), nc = std::min(p->nchans / 8 + 1, 8);
    PatternCost cost;
    int last = 0;                     // the tile before, and its cycles: straight lines between
    double before = 0;
    std::vector<uint8_t> len;
    try {
        for (int i = 0; i < nd; ++i) {
            const int t = nd > 1 ? (int)((int64_t)i * (ntiles - 1) / (nd - 1)) : 0;
            const int d0 = pattern_tile(ndm, ntiles, t);
            double tile = 0;
            for (int j = 0; j < nc; ++j) {
                const int c = (int)((2 * j + 1) * (int64_t)p->nchans / (2 * nc)) / 8 * 8;
                const int e = std::min(c + 8, p->nchans);
                const TileBuilder b(p, d0, pattern_tile(ndm, ntiles, t + 1) - d0, false, c, e);
                double cycles = 0;
                if (!b.cut(c, e, &len, &cycles)) return PatternCost{-1, 0};
                // (eight channels alone make 1.5% more of them than a whole tile's cut)
                tile += cycles / (e - c) / nc * p->nchans / 1.015;
            }
            cost.sum += tile + (t - last > 1 ? 0.5 * (t - last - 1) * (before + tile) : 0.0);
            cost.top = std::max(cost.top, tile);
            last = t;
            before = tile;
        }
    } catch (...) {
        return PatternCost{-1, 0};
    }
    return cost;
}

bool build_patterns(const hp_plan* p, DedispTiling* T) {
    const int ndm = p->ndm(), ntiles = (ndm + kPatBD - 1) / kPatBD;
    std::atomic<bool> failed{false};
    try {
        std::vector<DedispTiling> parts(ntiles);
        std::vector<double> cycles(ntiles, 0.0);
        // one thread per 1024 channels of a tile (about 0.5 ms)
        const int threads = (int)std::min<int64_t>((int64_t)ntiles * p->nchans / 1024, 16);
        const bool done = parallel_for(ntiles, threads, [&](int i) {
            if (failed) return;
            const int d0 = pattern_tile(ndm, ntiles, i), d1 = pattern_tile(ndm, ntiles, i + 1);
            TileOut out;
            for (int strict = 0; strict < 2 && !out.ok; ++strict) {
                out = TileOut();
                TileBuilder(p, d0, d1 - d0, strict != 0, 0, p->nchans).build(&out);
            }
            if (!out.ok) {
                failed = true;
                return;
            }
            DedispTiling& q = parts[i];
            q.tiles.push_back(TileDesc{d0, d1 - d0, 0, (int32_t)out.stages.size()});
            q.stages.swap(out.stages);
            q.chans.swap(out.chans);
            q.addr.swap(out.tab);
            q.max_reach = out.max_reach;
            cycles[i] = out.cost;
        });
        if (!done || failed) return false;
        append_tiling(parts, T);
        for (double c : cycles) {
            T->cost.sum += c;
            T->cost.top = std::max(T->cost.top, c);
        }
    } catch (...) {
        *T = DedispTiling();
        return false;
    }
    T->BD = kPatBD;
    T->BT = kPatBT;
    T->pattern = true;
    return true;
}

}  // namespace hp
