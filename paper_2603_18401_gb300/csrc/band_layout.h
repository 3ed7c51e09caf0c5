// Layout of the banded form's scratch (plain C++: no device code).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace egm {

// Angle buckets of the query order (egm_internal.cuh, query_bucket).
constexpr int kQSortBits = 11;
constexpr int kQBuckets = (1 << kQSortBits) + 2;
constexpr int kMaxSplit = 8;      // most items per tile of the banded form
constexpr int64_t kSplitItems = 4096;  // most items of a call with split tiles
constexpr int kQPlacePairs = 16;  // calls of up to so many pairs place the queries with several blocks a pair
constexpr int kBandTile = 128;    // queries per tile
constexpr int kBandRowBytes = 256;  // packed operand row
constexpr size_t kQueryRecBytes = 48;  // sizeof(QueryRec)

constexpr size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Banded-form scratch: query permutation and buckets; with float pairs
// (`packed`) also the sorted query records, the packed operand rows and
// their scales and norms (u8 and binary pairs' rows are read as they are).
// Without float pairs the operand buffers keep one tile of rows, which the
// band kernel's (unused) tensor maps cover.
//
// The query counts (qhist) lie first, at an offset and of a size that are the
// same for every call: the geometry kernel clears them while the previous
// call's last kernel may still run, on a layout of other sizes.  Bytes that
// no layout gives to anything else are safe to clear then, since the previous
// call's own counts are read before its band kernel starts.
struct BandLayout {
    size_t qhist, qperm, descA, descB, qbkt, qsrt, qscale, rnorm, fcand, fmask, qrank, part, part_n, arrived, total;
    int64_t items;
    BandLayout(int64_t nq, int64_t nr, int npairs, bool packed) {
        const size_t rb = (size_t)kBandRowBytes;
        const int64_t ta = packed ? nq : kBandTile, tb = packed ? nr : kBandTile;
        qhist = 0;
        qperm = qhist + align256(sizeof(uint32_t) * (size_t)kQBuckets * kQPlacePairs);
        descA = qperm + align256(sizeof(uint32_t) * (size_t)std::max<int64_t>(nq, 1));
        descB = descA + align256(rb * (size_t)std::max<int64_t>(ta, 1));
        qbkt = descB + align256(rb * (size_t)std::max<int64_t>(tb, 1));
        qsrt = qbkt + align256(sizeof(uint16_t) * (size_t)std::max<int64_t>(nq, 1));
        qscale = qsrt + align256(kQueryRecBytes * (size_t)std::max<int64_t>(packed ? nq : 1, 1));
        rnorm = qscale + align256(sizeof(float) * (size_t)std::max<int64_t>(packed ? nq : 1, 1));
        // 64 rows of padding: bulk copies of a 32-row box may run past the last row
        fcand = rnorm + align256(16 * (size_t)((packed ? nr : 0) + 64));
        fmask = fcand + align256(2 * 16 * (size_t)(packed ? nq : 0));
        qrank = fmask + align256(sizeof(uint32_t) * (size_t)(packed ? nq : 0));
        items = std::min<int64_t>(kMaxSplit * (nq / kBandTile + npairs), kSplitItems);
        part = qrank + align256(sizeof(uint32_t) * (size_t)std::max<int64_t>(nq, 1));
        part_n = part + align256(16 * (size_t)(items * kBandTile));
        arrived = part_n + align256(sizeof(uint32_t) * (size_t)(items * kBandTile));
        total = arrived + align256(sizeof(uint32_t) * (size_t)items);
    }
};

}  // namespace egm
