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
// computes [c0, c1), which holds what its own ranges of the later levels need.
// blk holds nt blocks of `stride` words (a multiple of 4):
//   header, level 0 (the source) .. nl: {c0, n, o0, o1}, n the computed rows |
//   the words of a row << 16, or on the columns axis the number of computed
//   groups of 4 columns | ceil(2^16 / that) << 8 (the source: its extent);
//   columns axis, level 1 .. nl, per group, 8 words: first words of the byte
//   pairs of outputs 0-1 and 2-3 (low, high half), their byte selectors, four
//   weight pairs (4096 - 2a | 2a << 16), 0, 0;
//   rows axis, level 1 .. nl, per row: (word offset of the source row << 16) | 2a.
// Source columns and rows count from the previous level's c0.
struct PyrAxis {
    int nt = 0, nl = 0, stride = 0;
    std::vector<int32_t> blk;
    std::vector<int32_t> extent;      // per level 0 .. nl: largest computed extent (pixels) of any tile
    int64_t computed = 0, owned = 0;  // pixels of levels 1 .. nl over all tiles
    bool ok = false;                  // source extents within max_extent, source steps within 3 columns
};
// sizes: extents of the source level and the nl levels.  row_words: null for the
// columns axis (16-byte aligned source, groups of 4), else per level 0 .. nl the
// words of a stored row (offsets stay below 2^16 words).
PyrAxis pyramid_axis(const int32_t* sizes, int nl, int nt, int max_extent, const int32_t* row_words = nullptr);
}  // namespace ofh
