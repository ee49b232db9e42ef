// rowshape.h -- how the row blocks (rowblock.cuh) cut a matrix up: lanes per row,
// units of rows, the lists of rows left to the second kernel and the pieces of
// very long rows.  Index arithmetic only, for host and device code alike.
// Row pointers are 32-bit with no more than 256 of headroom above the largest
// (SSSPMV_MAX_DIM), so no index is stepped by a piece (up to 2,048) before it
// is compared.
#pragma once
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define SSSPMV_HD __host__ __device__
#else
#define SSSPMV_HD
#endif

namespace ssspmv {

// shape of the row blocks, from m, nnz and the value type alone (so a batch and
// a single call agree on it, and with it on every sum's order)

struct RowShape {
    int32_t gs;     // log2 of the lanes per row
    int32_t us;     // log2 of the groups a warp takes at a time
    int32_t cap;    // most entries of a group that is staged
    int32_t piece;  // log2 of the entries of a piece of a very long row
};

// most entries a warp stages (the even split takes up to 31 per lane); at FP64
// 17 warps with stages this large leave 60 KB of L1
constexpr int32_t kStageMax = 888;

constexpr int32_t kMinCap = 640, kMinPiece = 10;

SSSPMV_HD inline RowShape row_shape(int32_t m, int32_t nnz, int32_t val_bytes)
{
    RowShape s;
    const int64_t mm = m > 0 ? m : 1;
    // one lane per row up to 27 entries on average (a 27-point stencil's 864
    // entries per group just fit), then 14 to 27 entries per lane; and more
    // lanes where the groups would be too few to keep every warp busy, if each
    // lane still gets enough entries: FP64 above 6 up to 1,024 groups, above 8
    // below 4,096.  Against 4 below 6,144 groups: bands, blocks and stencils of
    // 7,000 to 40,000 rows 9 to 11 us -> 7 to 9, R-MAT scale 16 27 to 29 -> 19
    // to 22 (the tiles: 25 to 27); whole groups from 1,536 on would make blocks
    // of 92 entries per row (27,000 rows) 18 us instead of 14.5 and rows of
    // 0..40 (120,007, axpby) 25.5 instead of 23.  In FP32 far fewer groups are
    // left whole, because the matrices of a batch share the GPU: 96 mixed ones
    // take 297 us below 384 groups, 317 below 1,536, 397 below 6,144, and
    // single small ones are as fast.
    s.gs = 0;
    while (s.gs < 5 && (int64_t)nnz > ((int64_t)27 << s.gs) * mm) ++s.gs;
    auto split = [&](int64_t below, int64_t entries) {
        return s.gs < 5 && (mm >> (5 - s.gs)) < below && (int64_t)nnz > (entries << s.gs) * mm;
    };
    while (val_bytes == 8 ? split(1025, 12) || split(4096, 16) : split(384, 8)) ++s.gs;
    // four groups at a time, where that leaves enough units for every warp
    // (half as many where several groups share a copy)
    const int64_t group = ((int64_t)nnz << (5 - s.gs)) / mm;  // its mean entries
    s.us = (mm >> (7 - s.gs)) >= (group <= 320 ? 3072 : 6144) ? 2 : 0;
    // room for groups well above the mean, and for several short ones
    int64_t cap = (group + group / 2) & ~(int64_t)7;
    if (cap < kMinCap) cap = kMinCap;
    if (cap > kStageMax) cap = kStageMax;
    s.cap = (int32_t)cap;
    // the lists have to fit the tiles' sections, which shrink per entry from
    // 15.7 million entries on (several tiles per bunch): twice as long pieces then
    s.piece = nnz <= 15000000 ? kMinPiece : kMinPiece + 1;
    return s;
}

// Most entries of a group that (r1) works off itself, a stage at a time; larger
// groups are listed.  Two stages, or, where a group is one row, as many as a
// warp's share of the matrix has, up to eight: rows that are all this long would
// nearly all be listed, a range of one row each or pieces of unlike lengths, and
// (r2) takes one such list entry per chain of loads.  50 million entries in rows
// of 2,100, two stages at most against this: FP64 197 us and 121 (the tiles 146),
// FP32 178 and 86 (90), BF16 values 176 and 81 (100); of 5,000: 158 and 118
// (165), 138 and 85 (111), 136 and 78 (100); of 900, two stages both times, but
// lane by lane now instead of split evenly: 180 and 143 (146), 133 and 100 (90),
// 133 and 99 (97).
SSSPMV_HD inline int32_t row_most(int32_t nnz, int32_t gs, int32_t cap)
{
    const int32_t share = nnz >> 12;
    if (gs < 5 || share <= 2 * cap) return 2 * cap;
    return share < 8 * cap ? share : 8 * cap;
}

// bounds of the lists (r1) writes, from groups of more than cap entries: at most
// one range of rows per `piece` entries or part of it of such a group, and rows
// longer than a piece cut into pieces
struct RowLists {
    int64_t ranges, pieces;
    size_t off_ranges, off_pieces, off_parts, off_arrived, bytes;  // from the lists' start
};

SSSPMV_HD inline RowLists row_lists(int64_t nnz, int32_t cap, int32_t piece)
{
    RowLists l;
    l.ranges = nnz / cap + (nnz >> piece) + 1;
    l.pieces = ((2 * nnz) >> piece) + 1;
    size_t o = 0;
    l.off_ranges = o;
    o = (o + 8 * (size_t)l.ranges + 15) & ~size_t(15);
    l.off_pieces = o;
    o = (o + 8 * (size_t)l.pieces + 15) & ~size_t(15);
    l.off_parts = o;
    o = (o + 8 * (size_t)l.pieces + 15) & ~size_t(15);
    l.off_arrived = o;
    l.bytes = o + 4 * (size_t)l.pieces;
    return l;
}

// units of rows of a matrix: three quarters of the rows in units of several
// groups, the rest one group each (they even out the end of the launch).  Some
// ten single groups per warp of the GPU are enough for that, two if they hold
// hardly any entries (means of up to 3): with a quarter of the rows of any
// matrix, 20 million rows of one entry were 273,000 units and 334 us, now
// 161,000 and 273 (FP32: 270 and 219), R-MAT scale 23 of edge factor 2 195 and
// 181; 2 million rows of one entry 30.6 and 27.5.
constexpr int32_t kMostSingles = 32768, kMostShortSingles = 6144;

struct RowUnits {
    int32_t nbig, nunits;
};

SSSPMV_HD inline RowUnits row_units(int32_t m, int32_t nnz, const RowShape &s)
{
    const int32_t rows = 32 >> s.gs, big_rows = rows << s.us;
    RowUnits u;
    int64_t big = (int64_t)m * 3 / 4;
    const int64_t singles = (int64_t)nnz <= 3 * (int64_t)m ? kMostShortSingles : kMostSingles;
    if (big < (int64_t)m - singles * rows) big = (int64_t)m - singles * rows;
    u.nbig = s.us > 0 ? (int32_t)(big / big_rows) : 0;
    u.nunits = u.nbig + (int32_t)(((int64_t)m - (int64_t)u.nbig * big_rows + rows - 1) / rows);
    return u;
}

// A row of more than 2^pl entries is cut into this many pieces of 2^pl, the
// last one shorter (or full); of no entries, none.
SSSPMV_HD inline int32_t row_pieces(int32_t len, int32_t pl)
{
    return len > 0 ? ((len - 1) >> pl) + 1 : 0;
}

// the end of the piece that starts at entry s of a row ending at e >= s
SSSPMV_HD inline int32_t piece_end(int32_t s, int32_t e, int32_t pl)
{
    return e - s > (1 << pl) ? s + (1 << pl) : e;
}

}  // namespace ssspmv
