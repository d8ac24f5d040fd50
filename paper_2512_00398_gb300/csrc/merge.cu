// merge.cu -- candidate merging and clustering on sm_103a (Section II-B,
// "Candidate Merging and Clustering"; Algorithm 1, last stage).
//
// Friends-of-friends over (trial, time window, width): two raw candidates are
// friends iff |d_i - d_j| <= dm_tol, |k_i - k_j| <= w_tol and their boxcar
// windows [t, t + W) lie within t_gap samples:
//   max(t_i, t_j) - min(t_i + W_i, t_j + W_j) <= t_gap.
// Clusters are connected components, so the result does not depend on the
// (atomic, unordered) order in which the detection kernel appended them.
//
//   1. keys (dm << 43 | sample << 5 | width) and exact sums S, padded with
//      UINT64_MAX; bitonic sort of 2048-key chunks in shared memory, then
//      merge passes that place every key by binary searches in the three partner
//      runs (keys are unique, so ranks are exact).
//   2. friends are linked by a lock-free union-find that always hangs the larger
//      root under the smaller one, so every root is the smallest index (= smallest
//      key) of its cluster.  With any width a friend's and t_gap >= 0 (the defaults),
//      the windows of one trial fall apart into components, in start order, wherever
//      a start lies more than t_gap past every end before it: a running maximum of
//      the ends finds them, and components of different trials are linked iff their
//      spans come within t_gap of each other.  (If a window q starts at most t_gap
//      after a component's end and ends at most t_gap before its start, take the
//      component's windows that start up to t_gap after q's end: the largest of their
//      ends is within t_gap of q's start, or the component would stop before q.)
//      Otherwise each candidate scans the windows that can touch its own.
//   3. per cluster: member count, trial and time ranges, and the member with
//      the largest S/N = S / (sigma * sqrt(W)), computed in FP64 with
//      correctly rounded operations (ties: smallest key).
//   4. roots are compacted in index order with a device-wide scan.
//
// A list of at most 1280 candidates (fewer with friend scans or a large dm_tol: small_list),
// the usual one, goes through all of it in one block's shared memory (merge_small_kernel); the
// kernels of the general path then find nothing to do.  The host cannot know the count,
// so they are launched all the same: few of them, and each starting while the one before
// it drains.
//
// Measured, against one union per touching pair, two-way passes and 21 launches: 215
// candidates (tiny search) 44 us, before 165; 25 855 (FAST-like file) 146, before
// 286; 3.4e7 in dense clusters (stress recipe, 2^20 samples) 20.0 ms, before 93.3, of
// which the pairwise links were 70.6; what is left there is the sort, 13 ms.
#include <algorithm>
#include <atomic>
#include <climits>

#include "common.cuh"

namespace hp {
namespace {

constexpr int kSortThreads = 1024;   // 2 keys per thread
constexpr uint64_t kPad = ~0ull;
// words of MergeArgs::scan: blocks of candidates handed out, CTAs done
constexpr int kLinkCounter = 0, kDoneCounter = 1, kMaxCounter = 2, kHeadCounter = 3;

__device__ __forceinline__ int key_dm(uint64_t k) { return (int)(k >> kKeyDmShift); }
__device__ __forceinline__ int64_t key_sample(uint64_t k) {
    return (int64_t)((k >> kKeySampleShift) & ((1ull << (kKeyDmShift - kKeySampleShift)) - 1));
}
__device__ __forceinline__ int key_width(uint64_t k) {
    return (int)(k & ((1u << kKeySampleShift) - 1));
}

__device__ __forceinline__ uint64_t cand_key(const hp_raw_cand& c) {
    return ((uint64_t)c.dm_idx << kKeyDmShift) | ((uint64_t)c.sample << kKeySampleShift) |
           (uint64_t)c.width_idx;
}

// The element-wise kernels walk the list with a grid stride: their grids are
// sized for the capacity only up to one resident wave, so a short list does not
// pay for tens of thousands of empty blocks.
#define FOR_EACH(i, n) \
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); \
         i += (int64_t)gridDim.x * blockDim.x)

// Bitonic sort of `size` (a power of two, at least 64) keys and their values in
// shared memory, one compare-exchange per thread and step; the steps inside a
// warp's 64 entries need no block barrier.
__device__ __forceinline__ void bitonic_sort(uint64_t* sk, int64_t* sv, int n) {
    const int t = threadIdx.x;
    const bool on = t < n / 2;
    for (int size = 2; size <= n; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (on) {
                const int i = (t / stride) * 2 * stride + t % stride, j = i + stride;
                const bool up = (i & size) == 0;
                const uint64_t ki = sk[i], kj = sk[j];
                if ((ki > kj) == up) {
                    sk[i] = kj;
                    sk[j] = ki;
                    const int64_t v = sv[i];
                    sv[i] = sv[j];
                    sv[j] = v;
                }
            }
            // the next step's pairs lie inside this warp's 64 entries too?
            if (stride > 32 || (stride == 1 && size >= 64)) __syncthreads(); else __syncwarp();
        }
    }
}

// Keys and sums of each chunk of 2048 candidates, sorted.
__global__ void __launch_bounds__(kSortThreads) chunk_sort_kernel(MergeArgs a) {
    __shared__ uint64_t sk[kSortChunk];
    __shared__ int64_t sv[kSortChunk];
    pdl_wait();
    const int64_t n = *a.n_clamped;
    // chunks blockIdx.x, blockIdx.x + gridDim.x, ... below n (block-uniform)
    for (int64_t base = (int64_t)blockIdx.x * kSortChunk; base < n;
         base += (int64_t)gridDim.x * kSortChunk) {
        for (int i = threadIdx.x; i < kSortChunk; i += blockDim.x) {
            sk[i] = kPad;
            sv[i] = 0;
            if (base + i < n) {
                const hp_raw_cand c = a.raw[base + i];
                sk[i] = cand_key(c);
                sv[i] = c.S;
            }
        }
        __syncthreads();
        bitonic_sort(sk, sv, kSortChunk);
        for (int i = threadIdx.x; i < kSortChunk; i += blockDim.x) {
            a.keys[0][base + i] = sk[i];
            a.vals[0][base + i] = sv[i];
        }
        __syncthreads();   // sk, sv are refilled with the next chunk
    }
}

// The buffer (0 or 1) that holds the sorted list of n after its merge passes.
__device__ __forceinline__ int sorted_in(int64_t n) {
    int c = 0;
    for (int64_t run = kSortChunk; run < n; run *= 4) c ^= 1;
    return c;
}

// Merge groups of four sorted runs: every key's rank is its place in its own run
// plus the keys below it in the other three.  A list that fits one run is in place.
__global__ void merge_pass_kernel(MergeArgs a, int64_t run, int from) {
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (run >= n) return;
    const uint64_t* __restrict__ ks = a.keys[from];
    FOR_EACH(i, n) {
        const int64_t r = i / run, g0 = (r & ~3ll) * run;
        const uint64_t key = ks[i];
        int64_t dst = g0 + (i - r * run);
#pragma unroll
        for (int64_t q = 1; q < 4; ++q) {
            const int64_t ps = (r ^ q) * run;
            if (ps >= n) continue;
            int64_t lo = ps, hi = min(ps + run, n);   // count partner keys < key
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (ks[mid] < key) lo = mid + 1; else hi = mid;
            }
            dst += lo - ps;
        }
        a.keys[from ^ 1][dst] = key;
        a.vals[from ^ 1][dst] = a.vals[from][i];
    }
}

__device__ __forceinline__ int32_t uf_find(int32_t* parent, int32_t x) {
    int32_t p = parent[x];
    while (p != x) {
        const int32_t g = parent[p];
        if (g != p) atomicCAS(&parent[x], p, g);   // path halving, keeps parent < child
        x = p;
        p = parent[x];
    }
    return x;
}

__device__ void uf_union(int32_t* parent, int32_t a, int32_t b) {
    while (true) {
        a = uf_find(parent, a);
        b = uf_find(parent, b);
        if (a == b) return;
        if (a > b) { const int32_t t = a; a = b; b = t; }
        if (atomicCAS(&parent[b], b, a) == b) return;   // b was still a root
    }
}

__device__ __forceinline__ int64_t lower_bound_key(const uint64_t* k, int64_t n, uint64_t key) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (k[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Union-find and cluster statistics before linking; trial_start[d] = the first
// sorted entry of trial d or later (d = ndm: n).
__global__ void link_init_kernel(MergeArgs a) {
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const uint64_t* keys = a.keys[sorted_in(n)];
    FOR_EACH(i, n) {
        a.parent[i] = (int32_t)i;
        a.best_bits[i] = 0;
        a.members[i] = 0;
        a.dm_lo[i] = INT_MAX;
        a.dm_hi[i] = INT_MIN;
        a.t_lo[i] = ~0ull;
        a.t_hi[i] = 0;
    }
    if (a.trial_start)
        FOR_EACH(d, (int64_t)a.ndm + 1)
            a.trial_start[d] = d == a.ndm ? n : lower_bound_key(keys, n, (uint64_t)d << kKeyDmShift);
}

// Is every pair of touching windows friends, whatever their widths (components)?
__host__ __device__ __forceinline__ bool any_window(const MergeArgs& a) {
    return a.w_tol >= a.nw - 1 && a.t_gap >= 0;
}

// Components: a candidate's trial and window end in one word, whose running maximum
// over the sorted list is the largest end so far in the candidate's own trial.
__device__ __forceinline__ uint64_t end_word(uint64_t key, const int32_t* widths) {
    return (key >> kKeyDmShift << kKeyDmShift) | (uint64_t)(key_sample(key) + widths[key_width(key)]);
}
constexpr uint64_t kEndMask = (1ull << kKeyDmShift) - 1;

// Does the candidate start a component, `before` being the running maximum before it?
__device__ __forceinline__ bool starts_component(uint64_t key, uint64_t before, int64_t t_gap) {
    return key >> kKeyDmShift != before >> kKeyDmShift ||
           key_sample(key) - (int64_t)(before & kEndMask) > t_gap;
}

// The component of one trial that ends with entry `last` (its first entry `head`)
// linked to those of the dm_tol trials after it.  Run(j): the running maximum up to
// entry j; head_of(j): the first entry of j's component.
template <class Run, class Head>
__device__ __forceinline__ void link_component(const MergeArgs& a, const uint64_t* keys, int64_t n,
                                               int64_t head, int64_t last, const Run& run,
                                               const Head& head_of, int32_t* parent,
                                               const int64_t* trial_start) {
    const int d = key_dm(keys[head]);
    const int64_t from = key_sample(keys[head]) - a.t_gap;            // ends from here on touch it
    const int64_t to = (int64_t)(run(last) & kEndMask) + a.t_gap;     // starts up to here do
    for (int dd = d + 1; dd <= d + a.dm_tol; ++dd) {
        int64_t b0, b1 = n;
        if (trial_start) {
            if (dd >= a.ndm) return;
            b0 = trial_start[dd];
            b1 = trial_start[dd + 1];
        } else {
            b0 = lower_bound_key(keys, n, (uint64_t)dd << kKeyDmShift);
            if (b0 >= n) return;
            const int next = key_dm(keys[b0]);
            if (next > dd) {        // no entry in trials dd .. next - 1
                dd = next - 1;
                continue;
            }
        }
        // the entries of trial dd that start at or before `to`, from the last one back
        // (`to` may lie past every sample that a key can hold)
        const uint64_t past = to + 1 < (int64_t)1 << (kKeyDmShift - kKeySampleShift)
                                  ? ((uint64_t)dd << kKeyDmShift) | ((uint64_t)(to + 1) << kKeySampleShift)
                                  : (uint64_t)(dd + 1) << kKeyDmShift;
        int64_t j = b0 + lower_bound_key(keys + b0, b1 - b0, past) - 1;
        while (j >= b0 && (int64_t)(run(j) & kEndMask) >= from) {
            const int64_t h = head_of(j);
            uf_union(parent, (int32_t)head, (int32_t)h);
            j = h - 1;
        }
    }
}

// Inclusive maximum over the warps of a 1024-thread block.
__device__ __forceinline__ uint64_t warp_max_scan(uint64_t x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t u = __shfl_up_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) >= o) x = max(x, u);
    }
    return x;
}

// Exclusive maximum of x over the 1024 threads of a block (0 before the first);
// total: over all of them.
__device__ __forceinline__ uint64_t block_max_exclusive(uint64_t x, uint64_t* warp_tot, uint64_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t incl = warp_max_scan(x);
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) warp_tot[lane] = warp_max_scan(warp_tot[lane]);
    __syncthreads();
    uint64_t before = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) before = 0;
    if (warp > 0) before = max(before, warp_tot[warp - 1]);
    *total = warp_tot[31];
    __syncthreads();   // warp_tot may be rewritten
    return before;
}

// The CTA that finishes last (of those that count themselves here) replaces v[0 ..
// count) by its exclusive maxima.  Every CTA calls it.
template <class T>
__device__ __forceinline__ void last_cta_max_scan(T* v, int64_t count, int32_t* done,
                                                  uint64_t* warp_tot) {
    __shared__ int32_t last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1) == (int32_t)gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    uint64_t carry = 0;
    for (int64_t b0 = 0; b0 < count; b0 += 1024) {
        const int64_t i = b0 + threadIdx.x;
        uint64_t total;
        const uint64_t x = i < count ? (uint64_t)__ldcg(&v[i]) : 0;
        const uint64_t e = max(carry, block_max_exclusive(x, warp_tot, &total));
        if (i < count) v[i] = (T)e;
        carry = max(carry, total);
    }
}

// The general path's component arrays, in buffers that are free between the sort
// and the statistics: the maximum of each chunk of 1024 end words (then before
// it), the running maxima, each entry's component head + 1 within its chunk (0: in
// a chunk before), the last head + 1 of each chunk (then before it).
struct Components {
    uint64_t* chunk_max;
    uint64_t* run;
    int32_t* head;
    int32_t* chunk_head;
    __device__ Components(const MergeArgs& a, int sorted)
        : chunk_max(a.keys[sorted ^ 1]), run(reinterpret_cast<uint64_t*>(a.vals[sorted ^ 1])),
          head(a.rep), chunk_head(a.block_sums) {}
    __device__ __forceinline__ int64_t head_of(int64_t i) const {
        const int32_t h = head[i];
        return (h > 0 ? h : chunk_head[i >> 10]) - 1;
    }
};

__global__ void __launch_bounds__(1024) chunk_max_kernel(MergeArgs a) {
    __shared__ uint64_t warp_tot[32];
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const int q = sorted_in(n);
    const Components C(a, q);
    const int64_t chunks = (n + 1023) / 1024;
    for (int64_t lb = blockIdx.x; lb < chunks; lb += gridDim.x) {
        const int64_t i = lb * 1024 + threadIdx.x;
        uint64_t total;
        block_max_exclusive(i < n ? end_word(a.keys[q][i], a.widths) : 0, warp_tot, &total);
        if (threadIdx.x == 0) C.chunk_max[lb] = total;
    }
    last_cta_max_scan(C.chunk_max, chunks, &a.scan[kMaxCounter], warp_tot);
}

__global__ void __launch_bounds__(1024) heads_kernel(MergeArgs a) {
    __shared__ uint64_t warp_tot[32];
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const int q = sorted_in(n);
    const Components C(a, q);
    const int64_t chunks = (n + 1023) / 1024;
    for (int64_t lb = blockIdx.x; lb < chunks; lb += gridDim.x) {
        const int64_t i = lb * 1024 + threadIdx.x;
        const uint64_t key = i < n ? a.keys[q][i] : 0;
        const uint64_t w = i < n ? end_word(key, a.widths) : 0;
        uint64_t total;
        const uint64_t before = max(C.chunk_max[lb], block_max_exclusive(w, warp_tot, &total));
        const bool head = i < n && (i == 0 || starts_component(key, before, a.t_gap));
        const uint64_t mine = head ? (uint64_t)(i + 1) : 0;
        const uint64_t h = max(mine, block_max_exclusive(mine, warp_tot, &total));
        if (i < n) {
            C.run[i] = max(before, w);
            C.head[i] = (int32_t)h;
        }
        if (threadIdx.x == 0) C.chunk_head[lb] = (int32_t)total;
    }
    last_cta_max_scan(C.chunk_head, chunks, &a.scan[kHeadCounter], warp_tot);
}

// Every entry under its component's head.
__global__ void attach_kernel(MergeArgs a) {
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const Components C(a, sorted_in(n));
    FOR_EACH(i, n) a.parent[i] = (int32_t)C.head_of(i);
}

// One component per thread that holds a component's last entry.
__global__ void link_components_kernel(MergeArgs a) {
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const int q = sorted_in(n);
    const Components C(a, q);
    FOR_EACH(i, n) {
        if (i + 1 < n && C.head[i + 1] != (int32_t)(i + 2)) continue;
        link_component(a, a.keys[q], n, C.head_of(i), i, [&](int64_t j) { return C.run[j]; },
                       [&](int64_t j) { return C.head_of(j); }, a.parent, a.trial_start);
    }
}

// Link candidate i to its friends j > i: in its own trial among the entries after
// it, in a later trial from the first entry at t_first (searched within that
// trial's entries when the per-trial table is there).
__device__ __forceinline__ void link_candidate(const MergeArgs& a, const int32_t* widths,
                                               const uint64_t* keys, int64_t n, int64_t i,
                                               int32_t* parent, const int64_t* trial_start) {
    const uint64_t ki = keys[i];
    const int di = key_dm(ki), wi = key_width(ki);
    const int64_t ti = key_sample(ki);
    const int64_t ei = ti + widths[wi];
    const int64_t t_first = ti - (int64_t)a.wmax - a.t_gap;
    const int64_t t_last = ei + a.t_gap;
    for (int dd = di; dd <= di + a.dm_tol; ++dd) {
        int64_t j0;
        if (dd == di) {
            j0 = i + 1;
        } else {
            const uint64_t lo_key = ((uint64_t)dd << kKeyDmShift) |
                                    ((uint64_t)(t_first > 0 ? t_first : 0) << kKeySampleShift);
            if (trial_start) {
                if (dd >= a.ndm) break;
                const int64_t b0 = trial_start[dd], b1 = trial_start[dd + 1];
                j0 = b0 + lower_bound_key(keys + b0, b1 - b0, lo_key);
            } else {
                j0 = lower_bound_key(keys, n, lo_key);
                if (j0 >= n) break;   // no later trial has an entry
            }
        }
        for (int64_t j = j0; j < n; ++j) {
            const uint64_t kj = keys[j];
            if (key_dm(kj) != dd) break;
            const int64_t tj = key_sample(kj);
            if (tj > t_last) break;
            const int wj = key_width(kj);
            if (abs(wi - wj) > a.w_tol) continue;
            const int64_t ej = tj + widths[wj];
            const int64_t gap = max(ti, tj) - min(ei, ej);
            if (gap <= a.t_gap) uf_union(parent, (int32_t)i, (int32_t)j);
        }
    }
}

// One candidate per thread, 256 at a time from a counter: the friend scans' work is
// heavy-tailed (dense clusters), and a fixed stride over one wave of blocks loses
// the balance (340 against 203 ms on 6.4e7 candidates); one block per 256 entries
// of the capacity keeps it but spends 57 us on empty blocks.
__global__ void __launch_bounds__(256) link_kernel(MergeArgs a) {
    __shared__ int32_t next;
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const uint64_t* keys = a.keys[sorted_in(n)];
    while (true) {
        if (threadIdx.x == 0) next = atomicAdd(&a.scan[kLinkCounter], 1);
        __syncthreads();
        const int64_t base = (int64_t)next * 256;
        __syncthreads();   // `next` is rewritten
        if (base >= n) return;
        const int64_t i = base + threadIdx.x;
        if (i < n) link_candidate(a, a.widths, keys, n, i, a.parent, a.trial_start);
    }
}

__device__ __forceinline__ double cand_snr(const MergeArgs& a, const int32_t* widths, uint64_t key,
                                           int64_t S) {
    if (a.sigw) return __ddiv_rn((double)S, a.sigw[(int64_t)key_dm(key) * a.nw + key_width(key)]);
    const double sg = a.sigma[key_dm(key)];
    const double sw = __dsqrt_rn((double)widths[key_width(key)]);
    return __ddiv_rn((double)S, __dmul_rn(sg, sw));
}

// Cluster statistics.  Neighbours in the sorted list are mostly of one cluster (the
// stress recipe's largest holds millions): a warp whose candidates all are adds
// them up first.
__global__ void stats_kernel(MergeArgs a) {
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const int c = sorted_in(n);
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i - (threadIdx.x & 31) < n; i += step) {
        const bool on = i < n;
        int32_t r = -1;
        unsigned long long best = 0, t0 = ~0ull, t1 = 0;
        int dm = 0;
        if (on) {
            r = uf_find(a.parent, (int32_t)i);
            a.parent[i] = r;   // (concurrent finds see a parent nearer the root)
            a.rep[i] = INT_MAX;
            const uint64_t k = a.keys[c][i];
            best = (unsigned long long)__double_as_longlong(cand_snr(a, a.widths, k, a.vals[c][i]));
            dm = key_dm(k);
            t0 = (unsigned long long)key_sample(k);
            t1 = t0 + (unsigned long long)a.widths[key_width(k)];
        }
        const int32_t r0 = __shfl_sync(0xffffffffu, r, 0);
        if (__all_sync(0xffffffffu, r == r0)) {   // (r0 >= 0: lane 0 is inside the list)
            const int lo = __reduce_min_sync(0xffffffffu, dm), hi = __reduce_max_sync(0xffffffffu, dm);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
                t0 = min(t0, __shfl_xor_sync(0xffffffffu, t0, o));
                t1 = max(t1, __shfl_xor_sync(0xffffffffu, t1, o));
            }
            if ((threadIdx.x & 31) == 0) {
                atomicMax(reinterpret_cast<unsigned long long*>(&a.best_bits[r]), best);
                atomicAdd(&a.members[r], 32);
                atomicMin(&a.dm_lo[r], lo);
                atomicMax(&a.dm_hi[r], hi);
                atomicMin(&a.t_lo[r], t0);
                atomicMax(&a.t_hi[r], t1);
            }
        } else if (on) {
            atomicMax(reinterpret_cast<unsigned long long*>(&a.best_bits[r]), best);
            atomicAdd(&a.members[r], 1);
            atomicMin(&a.dm_lo[r], dm);
            atomicMax(&a.dm_hi[r], dm);
            atomicMin(&a.t_lo[r], t0);
            atomicMax(&a.t_hi[r], t1);
        }
    }
}

// Exclusive scan of v over the 1024 threads of a block; total: their sum.
__device__ __forceinline__ int32_t block_exclusive(int32_t v, int32_t* warp_tot, int32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int32_t w = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        warp_tot[lane] = w;
    }
    __syncthreads();
    const int32_t before = warp > 0 ? warp_tot[warp - 1] : 0;
    *total = warp_tot[31];
    __syncthreads();   // warp_tot may be rewritten
    return before + x - v;
}

// Representatives, and the roots of every logical block of kScanBlock consecutive
// entries (each CTA takes logical blocks blockIdx.x, blockIdx.x + gridDim.x, ...);
// the CTA that finishes last scans the counts.
constexpr int kScanBlock = 1024;

__global__ void __launch_bounds__(kScanBlock) rep_count_kernel(MergeArgs a) {
    __shared__ int32_t cnt, last;
    __shared__ int32_t warp_tot[32];
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n < 0 || (n == 0 && blockIdx.x > 0)) return;
    const int c = sorted_in(n);
    const int64_t nblocks = (n + kScanBlock - 1) / kScanBlock;
    for (int64_t lb = blockIdx.x; lb < nblocks; lb += gridDim.x) {
        if (threadIdx.x == 0) cnt = 0;
        __syncthreads();
        const int64_t i = lb * kScanBlock + threadIdx.x;
        bool root = false;
        if (i < n) {
            const int32_t r = a.parent[i];
            root = r == (int32_t)i;
            const double snr = cand_snr(a, a.widths, a.keys[c][i], a.vals[c][i]);
            if ((unsigned long long)__double_as_longlong(snr) == (unsigned long long)a.best_bits[r])
                atomicMin(&a.rep[r], (int32_t)i);
        }
        const unsigned b = __ballot_sync(0xffffffffu, root);
        if ((threadIdx.x & 31) == 0 && b) atomicAdd(&cnt, __popc(b));
        __syncthreads();
        if (threadIdx.x == 0) a.block_sums[lb] = cnt;
        __syncthreads();   // cnt is cleared for the next logical block
    }
    if (threadIdx.x == 0) {
        __threadfence();
        const int32_t ctas = n == 0 ? 1 : (int32_t)gridDim.x;
        last = atomicAdd(&a.scan[kDoneCounter], 1) == ctas - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    int32_t carry = 0;
    for (int64_t b0 = 0; b0 < nblocks; b0 += 1024) {
        const int64_t i = b0 + threadIdx.x;
        int32_t total;
        const int32_t v = i < nblocks ? __ldcg(&a.block_sums[i]) : 0;
        const int32_t x = block_exclusive(v, warp_tot, &total);
        if (i < nblocks) a.block_sums[i] = carry + x;
        carry += total;
    }
    if (threadIdx.x == 0) *a.out_count = carry;
}

__global__ void __launch_bounds__(kScanBlock) scatter_kernel(MergeArgs a) {
    __shared__ int32_t warp_tot[32];
    pdl_wait();
    const int64_t n = *a.n_clamped;
    if (n <= 0) return;
    const int q = sorted_in(n);
    for (int64_t lb = blockIdx.x; lb * kScanBlock < n; lb += gridDim.x) {
        const int64_t i = lb * kScanBlock + threadIdx.x;
        const bool root = i < n && a.parent[i] == (int32_t)i;
        int32_t total;
        const int64_t slot = (int64_t)a.block_sums[lb] + block_exclusive(root, warp_tot, &total);
        if (!root || slot >= a.out_cap) continue;
        const int32_t rp = a.rep[i];
        const uint64_t kr = a.keys[q][rp];
        hp_cand c;
        c.dm_idx = key_dm(kr);
        c.width_idx = key_width(kr);
        c.sample = key_sample(kr);
        c.snr = (float)cand_snr(a, a.widths, kr, a.vals[q][rp]);
        c.members = a.members[i];
        c.dm_lo = a.dm_lo[i];
        c.dm_hi = a.dm_hi[i];
        c.t_lo = (int64_t)a.t_lo[i];
        c.t_hi = (int64_t)a.t_hi[i];
        a.out[slot] = c;
    }
}

// The whole merge of a short list in one block's shared memory; it leaves
// *n_clamped = -1 to the general path's kernels.  Longer lists: their length,
// the counters, the status.  What bounds it is the chain of barriers and
// shared-memory latencies of the sort (a list of 256 takes 3 block barriers, of
// 1024 13), the FP64 ratios (one each) and the links.
constexpr int kSmall = 1280;

// The longest list for one block, one candidate per thread up to 1024: up to here it is
// not slower than the general path's kernels on all 152 SMs.  Links to the next dm_tol
// trials grow with dm_tol, and one SM makes them; friend scans more so.  One block and
// general path, us, lists with clusters and dense ones:
//    defaults:           1030  71 and  89,  61 and 68       1400   90 and  83,   73 and  70
//    friend scans:       1030  94 and 126, 513 and 535      1400  137 and 125,  861 and 667
//    dm_tol 16:           768 140 and 132,  57 and 79       1536  345 and 151,   82 and  86
//    dm_tol 16, scans:    512 311 and 338, 508 and 622      1024  394 and 351,  986 and 1032
//    dm_tol 64:           256 159 and 254,  44 and 73       1024  615 and 291,   63 and  90
//    dm_tol 64, scans:    128 377 and 321, 146 and 339       512  863 and 581,  510 and 798
int64_t small_list(const MergeArgs& a) {
    const int reach = std::max(a.dm_tol, 1);
    return std::max(32, any_window(a) ? std::min(kSmall, 16384 / reach) : std::min(1088, 8192 / reach));
}

struct SmallState {
    uint64_t key[2048];            // (sorted as a power of two)
    int64_t val[2048];
    unsigned long long best[kSmall], t_lo[kSmall], t_hi[kSmall];
    int32_t parent[kSmall], rep[kSmall], members[kSmall], dm_lo[kSmall], dm_hi[kSmall];
    int32_t widths[kMaxWidths], warp_tot[32];
    uint64_t warp_max[32];
};

// Thread t holds the E entries from E t on of the list (n <= 1024 E).
template <int E>
__device__ __forceinline__ void merge_small(const MergeArgs& a, SmallState& s, int n) {
    const int i0 = E * (int)threadIdx.x;
    const int mine = min(E, n - i0);                 // entries of this thread (<= 0: none)
    uint64_t key[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        key[e] = 0;
        if (e < mine) {
            const int i = i0 + e;
            key[e] = s.key[i];
            s.best[i] = 0;
            s.members[i] = 0;
            s.dm_lo[i] = INT_MAX;
            s.dm_hi[i] = INT_MIN;
            s.t_lo[i] = ~0ull;
        }
    }
    if (any_window(a)) {
        // components: the running maxima in t_hi, the heads in parent
        uint64_t w[E], run = 0, total;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            w[e] = e < mine ? end_word(key[e], s.widths) : 0;
            run = max(run, w[e]);
        }
        run = block_max_exclusive(run, s.warp_max, &total);
        uint64_t h[E], last = 0;                     // head + 1 among this thread's entries
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (e < mine && (i0 + e == 0 || starts_component(key[e], run, a.t_gap)))
                last = (uint64_t)(i0 + e + 1);
            h[e] = last;
            run = max(run, w[e]);
            if (e < mine) s.t_hi[i0 + e] = run;
        }
        const uint64_t before = block_max_exclusive(last, s.warp_max, &total);
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e < mine) s.parent[i0 + e] = s.rep[i0 + e] = (int32_t)max(before, h[e]) - 1;
        __syncthreads();
        // (1024 apart: with neighbouring entries half of the threads had two and half none)
        for (int i = threadIdx.x; i < n; i += 1024)
            if (i + 1 == n || s.rep[i + 1] == i + 1)   // rep keeps the heads while parent changes
                link_component(a, s.key, n, s.rep[i], i, [&](int64_t j) { return (uint64_t)s.t_hi[j]; },
                               [&](int64_t j) { return (int64_t)s.rep[j]; }, s.parent, nullptr);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e < mine) s.parent[i0 + e] = i0 + e;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += 1024)
            link_candidate(a, s.widths, s.key, n, i, s.parent, nullptr);
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (e < mine) {
            s.rep[i0 + e] = INT_MAX;
            s.t_hi[i0 + e] = 0;
        }
    __syncthreads();
    double snr[E];
    int32_t root[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (e >= mine) continue;
        const uint64_t k = key[e];
        const int32_t r = root[e] = uf_find(s.parent, i0 + e);
        s.parent[i0 + e] = r;
        snr[e] = cand_snr(a, s.widths, k, s.val[i0 + e]);
        atomicMax(&s.best[r], (unsigned long long)__double_as_longlong(snr[e]));
        atomicAdd(&s.members[r], 1);
        atomicMin(&s.dm_lo[r], key_dm(k));
        atomicMax(&s.dm_hi[r], key_dm(k));
        const unsigned long long ts = (unsigned long long)key_sample(k);
        atomicMin(&s.t_lo[r], ts);
        atomicMax(&s.t_hi[r], ts + (unsigned long long)s.widths[key_width(k)]);
    }
    __syncthreads();
    int32_t roots = 0, total;
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (e < mine) {
            if ((unsigned long long)__double_as_longlong(snr[e]) == s.best[root[e]])
                atomicMin(&s.rep[root[e]], i0 + e);
            roots += root[e] == i0 + e;
        }
    int64_t slot = block_exclusive(roots, s.warp_tot, &total);   // (synchronises)
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = i0 + e;
        if (e >= mine || root[e] != i) continue;
        if (slot < a.out_cap) {
            const int32_t rp = s.rep[i];
            const uint64_t kr = s.key[rp];
            hp_cand c;
            c.dm_idx = key_dm(kr);
            c.width_idx = key_width(kr);
            c.sample = key_sample(kr);
            c.snr = (float)cand_snr(a, s.widths, kr, s.val[rp]);
            c.members = s.members[i];
            c.dm_lo = s.dm_lo[i];
            c.dm_hi = s.dm_hi[i];
            c.t_lo = (int64_t)s.t_lo[i];
            c.t_hi = (int64_t)s.t_hi[i];
            a.out[slot] = c;
        }
        ++slot;
    }
    if (threadIdx.x == 0) *a.out_count = total;
}

__global__ void __launch_bounds__(1024) merge_small_kernel(MergeArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    SmallState& s = *reinterpret_cast<SmallState*>(smem);
    const int t = threadIdx.x;
    pdl_wait();
    const int64_t nr = *a.nraw;
    const int64_t nc = nr < a.cap ? nr : a.cap;
    if (t == 0) {
        *a.n_clamped = nc <= a.small_max ? -1 : nc;
        if (nr > a.cap) latch_status(a.status, HP_ERR_CAND_OVERFLOW);
        if (nc > a.small_max)
            for (int i = 0; i < 4; ++i) a.scan[i] = 0;
    }
    if (nc > a.small_max) return;
    const int n = nc > 0 ? (int)nc : 0;
    int size = 64;
    while (size < n) size <<= 1;
    for (int i = t; i < size; i += 1024) {
        s.key[i] = kPad;
        s.val[i] = 0;
        if (i < n) {
            const hp_raw_cand c = a.raw[i];
            s.key[i] = cand_key(c);
            s.val[i] = c.S;
        }
    }
    if (t < a.nw) s.widths[t] = a.widths[t];
    __syncthreads();
    bitonic_sort(s.key, s.val, size);
    __syncthreads();
    if (n <= 1024)
        merge_small<1>(a, s, n);
    else
        merge_small<2>(a, s, n);
}

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// One resident wave of a strided kernel's blocks on the current device (its
// blocks per SM at full occupancy x the SM count), looked up once per kernel;
// a larger grid would leave a partial second wave with the same fixed share of
// work per thread.
template <class K>
int64_t wave(K kernel, int threads, std::atomic<int>& cache) {
    int v = cache.load(std::memory_order_relaxed);
    if (v == 0) {
        int dev = 0, sms = 0, per = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0) != cudaSuccess) {
            (void)cudaGetLastError();
            v = 1024;
        } else {
            v = std::max(1, sms * per);
        }
        cache.store(v, std::memory_order_relaxed);
    }
    return v;
}

std::atomic<int> g_wave[11];

}  // namespace

cudaError_t launch_merge(const MergeArgs& a_in, cudaStream_t s, int64_t* nlaunch) {
    MergeArgs a = a_in;
    a.small_max = small_list(a);
    if (a.cap <= 0) {
        return cudaMemsetAsync(a.out_count, 0, sizeof(int64_t), s);
    }
    cudaError_t e = cudaFuncSetAttribute(merge_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SmallState));
    if (e != cudaSuccess) return e;
    ++*nlaunch;
    e = launch_pdl(merge_small_kernel, 1, 1024, sizeof(SmallState), s, a);
    if (e != cudaSuccess || a.cap <= a.small_max) return e;
    const int64_t padded_cap = ceil_div(a.cap, kSortChunk) * kSortChunk;
    // grids of at most one resident wave; the kernels stride over the rest
    const int64_t g256 = ceil_div(padded_cap, 256);
    auto grid = [&](auto kernel, int threads, int64_t blocks, int id) {
        return (unsigned)std::min<int64_t>(blocks, wave(kernel, threads, g_wave[id]));
    };
    auto go = [&](cudaError_t r) {
        if (e == cudaSuccess) e = r;
        ++*nlaunch;
    };
    go(launch_pdl(chunk_sort_kernel, grid(chunk_sort_kernel, kSortThreads, padded_cap / kSortChunk, 0),
                  kSortThreads, 0, s, a));
    int from = 0;
    for (int64_t run = kSortChunk; run < a.cap; run *= 4, from ^= 1)
        go(launch_pdl(merge_pass_kernel, grid(merge_pass_kernel, 256, g256, 1), 256, 0, s, a, run, from));
    go(launch_pdl(link_init_kernel, grid(link_init_kernel, 256, std::max(g256, ceil_div((int64_t)a.ndm + 1, 256)), 2),
                  256, 0, s, a));
    const int64_t nblocks = ceil_div(padded_cap, kScanBlock);
    if (any_window(a)) {
        go(launch_pdl(chunk_max_kernel, grid(chunk_max_kernel, 1024, nblocks, 7), 1024, 0, s, a));
        go(launch_pdl(heads_kernel, grid(heads_kernel, 1024, nblocks, 8), 1024, 0, s, a));
        go(launch_pdl(attach_kernel, grid(attach_kernel, 256, g256, 9), 256, 0, s, a));
        go(launch_pdl(link_components_kernel, grid(link_components_kernel, 256, g256, 10), 256, 0, s, a));
    } else {
        go(launch_pdl(link_kernel, grid(link_kernel, 256, g256, 3), 256, 0, s, a));
    }
    go(launch_pdl(stats_kernel, grid(stats_kernel, 256, g256, 4), 256, 0, s, a));
    go(launch_pdl(rep_count_kernel, grid(rep_count_kernel, kScanBlock, nblocks, 5), kScanBlock, 0, s, a));
    go(launch_pdl(scatter_kernel, grid(scatter_kernel, kScanBlock, nblocks, 6), kScanBlock, 0, s, a));
    return e;
}

}  // namespace hp
