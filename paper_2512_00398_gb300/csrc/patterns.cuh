// patterns.cuh -- shapes and shared-memory table layout of the pattern-row
// dedispersion kernel (patterns.cu) and its host tiling (patterns.cpp).
#pragma once

#include <cstdint>

#include "hp_internal.h"

namespace hp {

// Trials per DM tile (4 summing warps x 6), packed words per trial and time
// tile: word i of a row holds samples i (low half) and i + kPatL (high half), so
// a time tile is 2 kPatL samples.
constexpr int kPatSumWarps = 4;
constexpr int kPatFormWarps = 11;
constexpr int kPatThreads = 32 * (kPatSumWarps + kPatFormWarps + 1);   // and one that copies
constexpr int kPatRD = 6;
constexpr int kPatBD = kPatSumWarps * kPatRD;
constexpr int kPatNJ = 32;               // words per lane and trial
constexpr int kPatL = 32 * kPatNJ;
constexpr int kPatBT = 2 * kPatL;
constexpr int kPatChunk = 128;           // words a warp forms per pattern at once
constexpr int kPatItem = 3;              // chunks of an item, a warp's unit of forming
constexpr int kPatMaxGroup = 4;          // channels summed into one pattern row
constexpr int kPatRowBufs = 2;           // ring of pattern-row buffers
constexpr int kPatRawBufs = 2;           // ring of staged bytes + set tables
constexpr int kPatTrialBufs = 4;         // ring of trial tables
constexpr int kPatRowBytes = 80 * 1024;
constexpr int kPatRawBytes = 30 * 1024;
constexpr int kPatTrialBytes = 1024;
constexpr int kPatPlaces = kPatRD <= 4 ? 4 : 8;   // trial table entries per summing warp
constexpr int kPatStageGroups = (kPatTrialBytes - 16) / (kPatSumWarps * kPatPlaces * 4);

// Form table of one stage, in the first kPatTabBytes of its raw buffer: this
// header, the items (warp w forms items begin[w] .. begin[w + 1] - 1), their rows.
constexpr int kPatTabBytes = 2048;
struct PatHeader {
    uint8_t begin[16];
};
static_assert(kPatFormWarps < 16, "PatHeader");
// Trial table: this header, then per group the byte offset in the row buffer of
// the first word that each of the kPatBD trials adds, kPatPlaces
// per summing warp (kPatRD of them used).
struct PatTrials {
    uint32_t ngroups;      // channel groups of the stage
    uint32_t flush;        // 1: add the 16-bit sums to the 32-bit sums after this stage
    uint32_t pad_[2];
};
// Patterns of one group whose channel offsets differ by at most their slot's shift
// (kPatShift1, kPatShift2) form a set: each channel's samples are unpacked once for all of them.  Channels
// sit in four slots (of a group of three the last is empty, of two the second and
// the last, of one the last three).  An item is 4 kPatItem words per lane of a set.
constexpr int kPatShift1 = 1, kPatShift2 = 2;   // of slot 1; of slots 2 and 3 (slot 0: none)
struct PatItem {
    uint32_t off[4];       // byte offset of each slot's first word in the raw buffer
    uint16_t row_off;      // byte offset of the item's rows in the table
    uint8_t nrows, nchan;  // rows, channels of the group
    uint16_t sel[4];       // PRMT selectors of each slot's first shift
    uint32_t pad_;
};
struct PatRow {
    uint32_t at;           // where the item's first chunk lies in the row buffer, + kPatItem - 1 chunks
    uint16_t put;          // bit e: the item's chunk e belongs to the row
    uint16_t kind;         // its shifts: slot 1's x 9 + slot 2's x 3 + slot 3's
};
static_assert(sizeof(PatHeader) == 16 && sizeof(PatTrials) == 16 && sizeof(PatItem) == 32 && sizeof(PatRow) == 8, "layout");

// A chunk's loads may start less than a chunk's bytes and one word before a row
// window and end as far behind it (what they form there is never added): the
// raw ring lies between the row buffers and the trial tables.
constexpr size_t kPatRawAt = (size_t)kPatRowBufs * kPatRowBytes;
constexpr size_t kPatTrialAt = kPatRawAt + (size_t)kPatRawBufs * kPatRawBytes;
constexpr size_t kPatSmem = kPatTrialAt + (size_t)kPatTrialBufs * kPatTrialBytes;
static_assert(kPatSmem + 512 <= 227 * 1024, "shared memory of one block");

}  // namespace hp
