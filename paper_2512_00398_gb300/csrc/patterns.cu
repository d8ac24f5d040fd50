// patterns.cu -- direct dedispersion from shared partial sums (Section II-B,
// "Incoherent Dedispersion"): the same exact sums as dedisp_rows_kernel with
// fewer additions.
//
// Within a tile of 24 neighbouring trials, the delays of four consecutive channels
// relative to the first of them (a pattern) take few distinct values: 4.9 on the
// 4096-channel, 1500-trial plan.  Each pattern is summed once into a row of 16-bit
// sums in shared memory, Q[u] = sum_k x_k[u + r_k], and every trial adds the row of
// its pattern at its own offset: one shared-memory word and one addition for two
// samples of four channels, against two words, four byte permutes and four
// additions for as many in the byte rows.
//
// A row's word i holds samples i and i + kPatL (not i and i + 1), so any offset is
// a whole number of words and adding a row needs no alignment; that costs two byte
// permutes per word when the row is formed, once per pattern.  Four warps add rows
// (6 trials x 32 words per lane fill their registers; the 32-bit sums live in
// tensor memory), eleven form them, one issues the bulk copies: with 8 + 7 warps of
// 3 trials it is 10% slower (the forming warps are bound by latency, so their number
// counts).  Registers are split by setmaxnreg,
// 4 x 224 + 12 x 96 per lane = the launch's 16 x 128.  Stages as large as shared
// memory allows (2.2 groups; two buffers of each kind) matter: the hand-over of a
// stage costs about 700 cycles, and three smaller buffers were 6-10% slower.
//
// What bounds it: latency and hand-overs, with the shared-memory pipe at 70% and
// the issue slots at 55% of their peaks; 1620 SM cycles per group of four channels,
// 24 trials and 2048 samples, of which adding the rows at one shared-memory
// wavefront per cycle would take 768.  Measured on the 4096-channel, 2^20-sample,
// 1500-trial file: 164.6 ms against 238.9 ms for the byte rows (35.7 against 24.6
// Tadd/s); 2048 channels, 2^18 samples, 750 trials: 10.7 against 14.5 ms.
#include <cstring>

#include "common.cuh"
#include "patterns.cuh"

namespace hp {
namespace {

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds8(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
// Predicated, without a branch between the chains that the two stores end.
__device__ __forceinline__ void sts128_if(uint32_t p, uint32_t a, uint32_t x, uint32_t y, uint32_t z,
                                          uint32_t w) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t"
        "@q st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w),
        "r"(p) : "memory");
}

// acc + x * m with m a runtime value: an IMAD, which the FMA pipe takes while the
// ALU pipe is busy with byte permutes.
__device__ __forceinline__ uint32_t imad(uint32_t x, uint32_t m, uint32_t acc) {
    uint32_t r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(m), "r"(acc));
    return r;
}

#define HP_R4(v, i) "=r"(v[i]), "=r"(v[i + 1]), "=r"(v[i + 2]), "=r"(v[i + 3])
#define HP_R16(v, i) HP_R4(v, i), HP_R4(v, i + 4), HP_R4(v, i + 8), HP_R4(v, i + 12)
#define HP_W4(v, i) "r"(v[i]), "r"(v[i + 1]), "r"(v[i + 2]), "r"(v[i + 3])

// 32 columns of the warp's 32 tensor-memory lanes (complete on return).
__device__ __forceinline__ void tmem_load32(uint32_t (&v)[32], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : HP_R16(v, 0), HP_R16(v, 16) : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// As above, 8 columns; the stores are complete after tmem_wait_stores.
__device__ __forceinline__ void tmem_load8(uint32_t (&v)[8], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : HP_R4(v, 0), HP_R4(v, 4) : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_store8(const uint32_t (&v)[8], uint32_t addr) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
        ::HP_W4(v, 0), HP_W4(v, 4), "r"(addr) : "memory");
}
__device__ __forceinline__ void tmem_wait_stores() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// A lane's NX consecutive samples of a channel from byte `sel` of the word at
// address at, with those kPatL later in the high halves.  Four samples at a time: one
// PRMT aligns the words, one takes two samples of each half (p = s0 + 2^8 s1 +
// 2^16 s0' + 2^24 s1'), one their odd bytes O, and p - 2^8 O are the even ones (the
// multiply-add keeps that off the ALU pipe).
template <int NX>
__device__ __forceinline__ void unpack(uint32_t (&x)[NX], uint32_t at, uint32_t sel, uint32_t m256) {
    constexpr int NWORDS = (NX + 6) / 4;   // the first sample is byte 0 .. 3 of the first word
    uint32_t w[NWORDS], h[NWORDS];
#pragma unroll
    for (int e = 0; e < NWORDS; ++e) {
        w[e] = lds32(at + 4 * e);
        h[e] = lds32(at + kPatL + 4 * e);
    }
#pragma unroll
    for (int e = 0; e < (NX + 2) / 4; ++e) {
        const uint32_t v = __byte_perm(w[e], w[e + 1], sel), u = __byte_perm(h[e], h[e + 1], sel);
        const uint32_t p01 = __byte_perm(v, u, 0x5410);
        x[4 * e + 1] = __byte_perm(p01, 0, 0x4341);
        x[4 * e] = imad(x[4 * e + 1], m256, p01);
        if (4 * e + 2 < NX) {
            const uint32_t p23 = __byte_perm(v, u, 0x7632);
            x[4 * e + 3] = __byte_perm(p23, 0, 0x4341);
            x[4 * e + 2] = imad(x[4 * e + 3], m256, p23);
        }
    }
    if constexpr (NX % 4 == 1) {   // one more: byte sel & 3 of the last word
        constexpr int e = NX / 4;
        x[NX - 1] = __byte_perm(w[e], h[e], (sel & 3u) * 0x101u + 0x400u) & 0x00FF00FFu;
    }
}

// a + b + c; volatile, so that the compiler does not merge the bodies of a switch
// into one that selects its operands at run time.
__device__ __forceinline__ uint32_t add3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm volatile("{\n\t.reg .u32 t;\n\tadd.u32 t, %1, %2;\n\tadd.u32 %0, t, %3;\n\t}"
                 : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// One row of an item: slots 0 and 1 (A), slot 2 shifted by S2 and slot 3 by S3.
template <int S2, int S3>
__device__ __forceinline__ void put_row(const uint32_t (&A)[4 * kPatItem],
                                        const uint32_t (&X2)[4 * kPatItem + kPatShift2],
                                        const uint32_t (&X3)[4 * kPatItem + kPatShift2], uint32_t to,
                                        uint32_t put, int lane) {
#pragma unroll
    for (int e = 0; e < kPatItem; ++e)   // (kPatItem lane + e) / 32: the chunk of those four words
        sts128_if(put >> ((uint32_t)(kPatItem * lane + e) >> 5) & 1u, to + (uint32_t)(16 * e),
                  add3(A[4 * e], X2[4 * e + S2], X3[4 * e + S3]),
                  add3(A[4 * e + 1], X2[4 * e + 1 + S2], X3[4 * e + 1 + S3]),
                  add3(A[4 * e + 2], X2[4 * e + 2 + S2], X3[4 * e + 2 + S3]),
                  add3(A[4 * e + 3], X2[4 * e + 3 + S2], X3[4 * e + 3 + S3]));
}

// One item: every slot's samples are unpacked once, over the shifts that occur in
// the set, so that a row is one three-input addition per word at offsets into
// them.  kPatItem is odd: lanes kPatItem words apart read 32 banks, and
// 16 kPatItem bytes apart store without conflicts.
__device__ __forceinline__ void form_item(uint32_t raw, uint32_t desc, uint32_t rows, int lane,
                                          uint32_t one) {
    static_assert(kPatItem % 2 == 1 && kPatChunk == 128, "bank conflicts; 32 lanes x 4 words");
    static_assert(kPatShift1 == 1 && kPatShift2 == 2, "the switch below");
    constexpr int N = 4 * kPatItem;
    const uint4 off = lds128(desc), S = lds128(desc + 16);
    const uint32_t m256 = one * 0xFFFFFF00u;
    const uint32_t at = raw + (uint32_t)(N * lane);
    const uint32_t nch = S.x >> 24;
    uint32_t A0[N], A1[N];
    {
        uint32_t X1[N + kPatShift1];
        unpack(A1, at + off.x, S.y, m256);
        unpack(X1, at + off.y, S.y >> 16, m256);
        if (nch < 3)
#pragma unroll
            for (int j = 0; j <= N; ++j) X1[j] = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            A0[j] = imad(A1[j], one, X1[j]);
            A1[j] = imad(A1[j], one, X1[j + 1]);
        }
    }
    uint32_t X2[N + kPatShift2], X3[N + kPatShift2];
    uint32_t tab = raw + (S.x & 0xFFFFu);
    const uint32_t end = tab + ((S.x >> 16) & 0xFFu) * (uint32_t)sizeof(PatRow);
    uint2 next = lds64(tab);
    unpack(X2, at + off.z, S.z, m256);
    unpack(X3, at + off.w, S.z >> 16, m256);
    if (nch < 4)
#pragma unroll
        for (int j = 0; j < N + kPatShift2; ++j) {
            X3[j] = 0;
            if (nch < 2) X2[j] = 0;
        }
    rows += (uint32_t)(16 * kPatItem * lane) - (uint32_t)((kPatItem - 1) * kPatChunk * 4);
#pragma unroll 1
    while (tab < end) {
        const uint32_t to = rows + next.x, put = next.y & 0xFFFFu, kind = next.y >> 16;
        tab += sizeof(PatRow);
        next = lds64(tab);   // after the last entry: inside the table's region
        switch (kind) {
#define HP_KIND(s2, s3)                                                            \
    case 3 * s2 + s3: put_row<s2, s3>(A0, X2, X3, to, put, lane); break;           \
    case 9 + 3 * s2 + s3: put_row<s2, s3>(A1, X2, X3, to, put, lane); break;
            HP_KIND(0, 0) HP_KIND(0, 1) HP_KIND(0, 2) HP_KIND(1, 0) HP_KIND(1, 1)
            HP_KIND(1, 2) HP_KIND(2, 0) HP_KIND(2, 1) HP_KIND(2, 2)
#undef HP_KIND
        }
    }
}

// Add the rows of G groups (trial tables at tab, one group after the other) to
// the warp's trials, eight words of each row at a time: the next eight are loaded
// before the last eight are added, since one warp per scheduler has nothing else
// to hide the loads behind.
template <int G>
__device__ __forceinline__ void add_rows(uint32_t (&acc)[kPatRD][kPatNJ], uint32_t rows,
                                         uint32_t tab) {
    constexpr int B = 8, NB = kPatNJ / B;
    uint32_t at[2][G], v[2][G][B];
#pragma unroll
    for (int g = 0; g < G; ++g) at[0][g] = rows + lds32(tab + (uint32_t)(g * kPatSumWarps * kPatPlaces * 4));
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int j = 0; j < B; ++j) v[0][g][j] = lds32(at[0][g] + 128 * j);
#pragma unroll
    for (int i = 0; i < kPatRD * NB; ++i) {
        const int r = i / NB, j0 = (i % NB) * B, n = i + 1;
        if (i % NB == 0 && r + 1 < kPatRD)
#pragma unroll
            for (int g = 0; g < G; ++g)
                at[(r + 1) & 1][g] = rows + lds32(tab + (uint32_t)(g * kPatSumWarps * kPatPlaces * 4 + 4 * (r + 1)));
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if (n < kPatRD * NB)
#pragma unroll
                for (int g = 0; g < G; ++g)
                    v[n & 1][g][j] = lds32(at[(n / NB) & 1][g] + 128 * ((n % NB) * B + j));
            // (volatile: in this order between the loads, not after them)
            if constexpr (G == 2)
                acc[r][j0 + j] = add3(acc[r][j0 + j], v[i & 1][0][j], v[i & 1][1][j]);
            else
                asm volatile("add.u32 %0, %0, %1;" : "+r"(acc[r][j0 + j]) : "r"(v[i & 1][0][j]));
        }
    }
}

// SPLIT: tiles of jobs with J.pattern > 1 are shared by that many blocks, each with a part
// of the stages, whose sums are added to the zeroed output (plan.cpp, pattern_waves, has
// when and the figures).
// Warps 0-3 add pattern rows (six trials of the tile each), warps 4-14 form them
// from the staged bytes, warp 15 issues the bulk copies.  The summing warps hold
// six trials x 32 packed words per lane; their 32-bit sums are in tensor memory
// (48 K words), where the 16-bit sums are added every 256 channels.
template <bool SPLIT>
__global__ void __launch_bounds__(kPatThreads, 1)
dedisp_patterns_kernel(const __grid_constant__ DedispBatch batch, int* status, uint64_t timeout_ns,
                       uint32_t one) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ uint64_t raw_full[kPatRawBufs], raw_free[kPatRawBufs];
    __shared__ uint64_t formed[kPatRowBufs], row_free[kPatRowBufs];
    __shared__ int abort_flag;
    __shared__ int issued;                  // stages whose copies were issued
    __shared__ uint32_t tmem_base;
    const uint32_t rows0 = smem_u32(smem);
    const uint32_t raw0 = rows0 + (uint32_t)kPatRawAt, trial0 = rows0 + (uint32_t)kPatTrialAt;

    const int64_t blk = blockIdx.x;
    int jb = 0;
    while (jb + 1 < batch.njobs && batch.prefix[jb + 1] <= blk) ++jb;
    const DedispJob& J = batch.jobs[jb];
    // groups of eight time tiles, every DM tile of a group before the next group
    // (the windows of a group's rows stay in L2)
    constexpr int TG = 8;
    // (a tile of a split job belongs to J.pattern blocks, each with a part of its stages)
    const int nparts = SPLIT ? (int)J.pattern : 1;
    const int64_t item = (blk - batch.prefix[jb]) / nparts;
    const int64_t per = (int64_t)TG * J.ndt;
    const int64_t grp = item / per;
    const int64_t rem = item - grp * per;
    const int64_t gsz = min((int64_t)TG, (int64_t)J.ntt - grp * TG);
    const int dt = (int)(rem / gsz);
    const int tt = (int)(grp * TG + rem % gsz);
    TileDesc T = J.tiles[dt];
    if (SPLIT && nparts > 1) {
        const int part = (int)((blk - batch.prefix[jb]) % nparts);
        const int s0 = T.nstages * part / nparts, s1 = T.nstages * (part + 1) / nparts;
        if (s0 == s1) return;                                  // the whole block
        T.stage_begin += s0;
        T.nstages = s1 - s0;
    }
    const int64_t t0 = (int64_t)tt * kPatBT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nst = T.nstages;
    static_assert(kPatTrialBufs >= kPatRawBufs + kPatRowBufs, "trial slots outlive their stage");

    if (tid == 0) {
        for (int b = 0; b < kPatRawBufs; ++b) {
            mbar_init(&raw_full[b], 1);
            mbar_init(&raw_free[b], kPatFormWarps);
        }
        for (int b = 0; b < kPatRowBufs; ++b) {
            mbar_init(&formed[b], kPatFormWarps);
            mbar_init(&row_free[b], kPatSumWarps);
        }
        mbar_fence_init();
        abort_flag = 0;
        issued = 0;
    }
    if (warp == 0) {
        // all 512 columns: one block per SM (shared memory), no other user
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                         smem_u32(&tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    volatile int* abort = &abort_flag;
    // The n-th phase of a barrier, warp-uniform: one try that may suspend the warp
    // for up to 20 us before the clock and the abort flag are polled.
    auto wait = [&](uint64_t* bar, int n) -> bool {
        const uint32_t parity = (uint32_t)n & 1u;
        const bool ok = mbar_try_wait_suspended(bar, parity, 20000) ||
                        mbar_wait_or_abort(bar, parity, timeout_ns, abort);
        return __all_sync(0xffffffffu, ok);
    };

    if (warp >= kPatSumWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 96;");
        if (warp == kPatSumWarps + kPatFormWarps) {
            // Bulk copies of every stage: its set table and the channel rows' windows
            // into a raw buffer once stage s - 2 is formed, its trial table into the slot
            // of stage s - 4, which was summed before stage s - 2 could be formed.  A
            // stage's row descriptors are read a stage ahead, the stage descriptors that
            // name them two: two dependent reads from global memory take longer than a
            // stage.
            const StageDesc* stages = J.stages + T.stage_begin;
            const ChanDesc* chans = J.chans;
            StageDesc S = stages[0], S1 = stages[min(1, nst - 1)];
            ChanDesc cd = chans[S.chan_begin + min((uint32_t)lane, S.nchan - 1)];
            for (int s = 0; s < nst; ++s) {
                const int b = s % kPatRawBufs, tb = s % kPatTrialBufs;
                const StageDesc S2 = stages[min(s + 2, nst - 1)];
                const ChanDesc cd1 = chans[S1.chan_begin + min((uint32_t)lane, S1.nchan - 1)];
                if (s >= kPatRawBufs && !wait(&raw_free[b], s / kPatRawBufs - 1)) break;
                uint8_t* B = smem + kPatRawAt + b * kPatRawBytes;
                if (lane == 0) {
                    issued = s + 1;
                    mbar_arrive_expect_tx(&raw_full[b], S.tx_bytes);
                    bulk_copy_g2s(smem + kPatTrialAt + tb * kPatTrialBytes,
                                  J.addr + S.addr_begin + S.addr_bytes / 4, S.addr_off,
                                  &raw_full[b]);
                    bulk_copy_g2s(B, J.addr + S.addr_begin, S.addr_bytes, &raw_full[b]);
                }
                __syncwarp();
                if (lane < S.nchan)
                    bulk_copy_g2s(B + cd.offB, J.xt + (int64_t)cd.c * J.xt_pitch + t0 + cd.goff,
                                  4 * cd.nwords, &raw_full[b]);
                S = S1;
                S1 = S2;
                cd = cd1;
            }
        } else {
            const uint32_t fw = (uint32_t)(warp - kPatSumWarps);
            for (int s = 0; s < nst; ++s) {
                const int b = s % kPatRawBufs, rb = s % kPatRowBufs;
                if (!wait(&raw_full[b], s / kPatRawBufs)) break;
                if (s >= kPatRowBufs && !wait(&row_free[rb], s / kPatRowBufs - 1)) break;
                const uint32_t raw = raw0 + (uint32_t)(b * kPatRawBytes);
                const uint32_t rows = rows0 + (uint32_t)(rb * kPatRowBytes);
                const uint32_t begin = lds8(raw + fw), end = lds8(raw + fw + 1);
#pragma unroll 1
                for (uint32_t i = begin; i < end; ++i)
                    form_item(raw, raw + 16 + 32 * i, rows, lane, one);
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&formed[rb]);
                    mbar_arrive(&raw_free[b]);
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        uint32_t acc[kPatRD][kPatNJ];
#pragma unroll
        for (int r = 0; r < kPatRD; ++r)
#pragma unroll
            for (int j = 0; j < kPatNJ; ++j) acc[r][j] = 0;
        // this warp's 32 lanes x 256 columns of tensor memory: the 32-bit sums
        const uint32_t tmem = tmem_base + ((uint32_t)(warp & 3) << 21) +
                              (uint32_t)(warp >> 2) * (2 * kPatRD * kPatNJ);
        bool first = true, ok = true;
        for (int s = 0; s < nst; ++s) {
            const int tb = s % kPatTrialBufs, rb = s % kPatRowBufs;
            // (the forming warps had waited for the stage's copies, its trial table among them)
            if (!(ok = wait(&formed[rb], s / kPatRowBufs))) break;
            const uint32_t rows = rows0 + (uint32_t)(rb * kPatRowBytes) + 4u * (uint32_t)lane;
            uint32_t tab = trial0 + (uint32_t)(tb * kPatTrialBytes);
            const uint2 H = lds64(tab);
            tab += 16 + (uint32_t)(warp * kPatPlaces * 4);
            uint32_t g = warp * kPatRD < T.nd ? H.x : 0;
            for (; g >= 2; g -= 2, tab += 2 * kPatSumWarps * kPatPlaces * 4) add_rows<2>(acc, rows, tab);
            if (g) add_rows<1>(acc, rows, tab);
            __syncwarp();
            if (lane == 0) mbar_arrive(&row_free[rb]);
            if (H.y || (SPLIT && s == nst - 1)) {   // add the 16-bit sums to the 32-bit sums
#pragma unroll
                for (int r = 0; r < kPatRD; ++r)
#pragma unroll
                    for (int e = 0; e < kPatNJ / 4; ++e) {
                        const int half = e / (kPatNJ / 8), j0 = e % (kPatNJ / 8) * 8;
                        const uint32_t at = tmem + (uint32_t)((2 * r + half) * kPatNJ + j0);
                        uint32_t v[8];
                        if (first) {
#pragma unroll
                            for (int j = 0; j < 8; ++j) v[j] = 0;
                        } else {
                            tmem_load8(v, at);
                        }
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            v[j] += half ? acc[r][j0 + j] >> 16 : acc[r][j0 + j] & 0xFFFFu;
                        tmem_store8(v, at);
                    }
                tmem_wait_stores();
#pragma unroll
                for (int r = 0; r < kPatRD; ++r)
#pragma unroll
                    for (int j = 0; j < kPatNJ; ++j) acc[r][j] = 0;
                first = false;
            }
        }
        if (ok) {
#pragma unroll 1
            for (int r = 0; r < kPatRD; ++r) {
                const int dl = warp * kPatRD + r;
                if (dl >= T.nd) break;
                int32_t* row = J.out + (int64_t)(T.d0 + dl) * J.out_pitch;
#pragma unroll 1
                for (int e = 0; e < 2; ++e) {
                    uint32_t v[kPatNJ];
                    tmem_load32(v, tmem + (uint32_t)((2 * r + e) * kPatNJ));
#pragma unroll
                    for (int j = 0; j < kPatNJ; ++j) {
                        const int64_t t = t0 + e * kPatL + 32 * j + lane;
                        if (t < J.nout) {
                            if (!SPLIT || nparts == 1)
                                row[t] = (int32_t)v[j];
                            else                               // (zeroed before the launch)
                                atomicAdd(&row[t], (int32_t)v[j]);
                        }
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();   // every warp comes here (each wait is bounded)
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0 && *abort) {
        latch_status(status, HP_ERR_TIMEOUT);
        // only the last kPatRawBufs issued stages can still be in flight
        for (int x = issued > kPatRawBufs ? issued - kPatRawBufs : 0; x < issued; ++x)
            mbar_wait_bounded(&raw_full[x % kPatRawBufs], (uint32_t)(x / kPatRawBufs) & 1u, timeout_ns);
    }
    __syncwarp();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base));
}

}  // namespace

cudaError_t launch_dedisp_patterns(const DedispBatch& b, int* status, uint64_t timeout_ns,
                                   cudaStream_t s) {
    const int64_t total = b.prefix[b.njobs];
    if (total <= 0) return cudaSuccess;
    // (the kernel without the parts of tiles is 1 to 2% faster)
    bool split = false;
    for (int j = 0; j < b.njobs; ++j) split = split || b.jobs[j].pattern > 1;
    const auto k = split ? dedisp_patterns_kernel<true> : dedisp_patterns_kernel<false>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kPatSmem);
    if (e != cudaSuccess) return e;
    k<<<(unsigned)total, kPatThreads, kPatSmem, s>>>(b, status, timeout_ns, 1u);
    return cudaGetLastError();
}

}  // namespace hp
