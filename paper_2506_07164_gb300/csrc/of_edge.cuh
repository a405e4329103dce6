// Wide loads at the end of a caller's frame.
//
// A frame of pitch p holds (h - 1) p + w bytes: the padding behind its last row
// may belong to something else, or to nothing.  Kernels that read a frame's
// bytes in aligned words take the word that would pass this end bytewise.
#pragma once
#include <cuda_runtime.h>

namespace ofk {

// Columns x - H .. x + H of rows y - H .. y + H of a w x h image as aligned
// words, `row_words` places a row: place i is word i % row_words (< nw) of row
// i / row_words.  The places below `whole` may be read as words; with `tail`,
// place `whole` is the last word of the last row and passes the frame's end.
struct PatchWords {
    int sh, nw, whole;
    bool tail;
};
__host__ __device__ __forceinline__ PatchWords patch_words(int x, int y, int H, int w, int h, int row_words) {
    PatchWords p;
    p.sh = (x - H) & 3;
    p.nw = (p.sh + 2 * H + 4) >> 2;
    p.tail = y + H == h - 1 && x - H - p.sh + 4 * p.nw > w;
    p.whole = 2 * H * row_words + p.nw - (p.tail ? 1 : 0);
    return p;
}

// Of the 16 bytes from column x of row y (both inside a w x h image), those
// inside the row; whether they may be read as one 16-byte load.
__host__ __device__ __forceinline__ int chunk_bytes(int x, int w) { return w - x < 16 ? w - x : 16; }
__host__ __device__ __forceinline__ bool chunk_whole(int n, int y, int h) { return n == 16 || y < h - 1; }

}  // namespace ofk
