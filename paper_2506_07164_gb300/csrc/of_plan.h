// Host-side plan arithmetic (of_plan.cpp).
#pragma once
#include <stdint.h>

#include <vector>

namespace ofh {
void level_sizes(int W, int H, int levels, float scale, int32_t* ws, int32_t* hs, double* ls);
void level_quotas(int N, int L, float scale, int32_t* q);
void resize_table(int n_src, int n_dst, int32_t* tab);
bool k_fraction(float k, int64_t* num, int64_t* den);
// (1 / (4*7*255))^4 / den as float: the keypoint response is key * this
// (float arithmetic; within 3e-7 relative of the float64 quotient).
float response_scale(int64_t den);

// One axis of a fused run of pyramid levels (k_pyramid): nl levels computed
// from a source level by nt tiles.  Tile i owns [o0, o1) of every level and
// computes [c0, c1), which holds what its own ranges of the later levels need
// (columns: from a multiple of 16 of the source, in groups of 4 of the levels).
// Its tables are nt blocks of `stride` words (a multiple of 4):
//   header, level 0 (the source) .. nl: {c0, n, o0, o1}, n the computed rows |
//   the words of a row << 16, or on the columns axis the number of computed
//   groups of 4 columns | ceil(2^16 / that) << 8 (the source: its extent);
//   columns axis, level 1 .. nl, per group, 8 words: first words of the byte
//   pairs of outputs 0-1 and 2-3 (low, high half), their byte selectors, four
//   weight pairs (4096 - 2a | 2a << 16), 0, 0;
//   rows axis, level 1 .. nl, per row: (word offset of the source row << 16) | 2a
//   (offsets stay below 2^16 words).
// Source columns and rows count from the previous level's c0.
struct PyrRange {
    int32_t c0 = 0, c1 = 0, o0 = 0, o1 = 0;
};
struct PyrAxis {
    int nt = 0, nl = 0, stride = 0;
    std::vector<PyrRange> ranges;     // nt tiles of nl + 1 levels
    std::vector<int32_t> extent;      // per level 0 .. nl: largest computed extent (pixels) of any tile
    int64_t computed = 0, owned = 0;  // pixels of levels 1 .. nl over all tiles
    bool ok = false;                  // source extents within max_extent
};

// A frame's levels as runs of at most max_levels levels, each of as many as keep
// the seams (computed over owned pixels) within max_seam at the largest tile of
// the source level that fits, starting from `tile` pixels a side.  ws, hs: the
// levels' sizes; xtab[l], ytab[l], l >= 1: the resize tables from level l - 1.
// False: some level's source steps (above 3 columns) or pieces do not fit.
// Planning a shape is part of the first call with it, so the search compares
// ranges, a few numbers per tile and level, and only the chosen runs get their
// tables (pyramid_tables).
struct PyrPiece {
    int level = 0, nl = 0, ntx = 0, nty = 0;
    PyrAxis x, y;
};
bool pyramid_pieces(const std::vector<int32_t>& ws, const std::vector<int32_t>& hs, const std::vector<const int32_t*>& xtab,
                    const std::vector<const int32_t*>& ytab, int max_levels, int tile, double max_seam,
                    std::vector<PyrPiece>& out);
// A run's column and row tables: x.stride * x.nt and y.stride * y.nt words, zero before.
void pyramid_tables(const PyrPiece& p, const std::vector<int32_t>& ws, const std::vector<int32_t>& hs,
                    const std::vector<const int32_t*>& xtab, const std::vector<const int32_t*>& ytab, int32_t* x, int32_t* y);
}  // namespace ofh
