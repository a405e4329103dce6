// Orientation by intensity centroid (Fig. 1 "Centroid") and the output
// records.  One warp per output slot (frame, level, rank):
//   - the keypoint's patch (31 x 31 for radius 15) goes to shared memory as
//     aligned words, 9 loads per lane in flight at once;
//   - lane = column u: moments m10 = sum u I, m01 = sum v I over the disc
//     u^2 + v^2 <= r^2 from the column's sums, warp reduction;
//   - Harris sums A, B, C of the kept keypoint (Eqs. 2-4): lanes hold columns,
//     so the vertical Sobel passes are a lane's own rows and the horizontal
//     ones two shuffles per row, warp reduction;
//   - angle = atan2f(m01, m10) (both moments are exact int32, |m| < 2^24, so
//     their float conversion is exact);
//   - response = key / kden * (1 / (4*7*255))^4, as key (float) times the
//     host-rounded float (1/(4*7*255))^4 / kden (relative error below 3e-7);
//   - level-0 coordinates from the plan's tables (x * scale^level rounded once).
//   - rank: the list's own order, or (GROUPED) of a list grouped by key code,
//     better codes first, the start of the code's run plus the better ones of the
//     run (key descending, then y, then x ascending); the 32 entries around the
//     keypoint usually hold the run, and are read beside its patch.
// Records are level-major in rank order: the place of a kept keypoint is the
// number of keypoints kept by the frame's earlier levels plus its rank.
//
// Bound by the latency of a warp's chain of loads (descriptors, position,
// pixels), so each link is one round: the counts of the earlier levels by one
// lane each, everything that depends on the position together.  128 1080p frames
// (128 k keypoints): 145 us with byte loads in rounds of 8, two rounds of Sobel
// loads and the counts and the score one after another, 108 us now, bound by
// instruction issue (70 %).
#include <cuda_runtime.h>

#include "of_edge.cuh"
#include "of_internal.h"
#include "of_launch.cuh"
#include "of_rank.cuh"

namespace ofk {

constexpr int OP_WORDS = 9;                   // aligned words that hold any 31 bytes
constexpr int OP_SIZE = 31 * OP_WORDS;        // words of a patch

template <bool GROUPED, bool SPARSE>
__global__ void __launch_bounds__(ORIENT_WARPS * 32)
k_orient(const Img* __restrict__ imgs, int img_begin, int n_img, int slot_begin, int slot_end,
         const Call* __restrict__ call, const uint16_t* __restrict__ slot_img) {
    __shared__ uint32_t patch[ORIENT_WARPS][OP_SIZE];
    const int slot = slot_begin + blockIdx.x * ORIENT_WARPS + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_trigger();
    if (slot >= slot_end) {
        pdl_wait();
        return;
    }
    // The slot's image: from the plan's slot table, else a search over slot0.
    int lo = img_begin, hi = img_begin + n_img - 1;
    if (slot_img) {
        lo = __ldg(slot_img + slot);
    } else {
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (imgs[mid].slot0 <= slot) lo = mid; else hi = mid - 1;
        }
    }
    const Img& I = imgs[lo];
    const int idx = slot - I.slot0;  // the keypoint in the image's list
    const int levels = call->levels, n_features = call->n_features;
    const int quota = I.quota, frame = I.frame;
    const int32_t* const ctr = I.ctr;
    if (SPARSE) {
        // More slots than the images can be expected to fill: those beyond their list go
        // before the rest is read (96 160 x 120 frames of 8192 features, whole call 151 us
        // otherwise, 132 so; with full lists the later reads would cost 4 % of this kernel).
        pdl_wait();
        if (slot != frame * n_features && (idx >= quota || idx >= ctr[1])) {
            pdl_wait();  // long over: every exit stands directly behind a wait
            return;
        }
    }
    // Descriptor fields, read before the wait; lane l < levels: level l's counters.
    const uint8_t* const img = I.img;
    const uint8_t* const score = I.score;
    const float* const fx = I.fx;
    const float* const fy = I.fy;
    const int pitch = I.pitch, spitch = I.spitch, level = I.level;
    const int width = I.w, height = I.h;
    const int32_t* const lctr = lane < levels ? imgs[frame * levels + lane].ctr : nullptr;
    const uint32_t* const kyx = I.kyx;
    const uint64_t* const kkey = I.kkey;
    const int R = call->radius, H = max(R, 4);  // H: rows and columns around the keypoint that are read
    pdl_wait();  // the kept keypoints
    if (idx >= quota && slot != frame * n_features) return;
    const int kept_l = lctr ? lctr[1] : 0;
    const int kept = ctr[1];
    // The keypoint's entry (GROUPED: the 32 around it, itself in lane 16), issued beside
    // the counts; unused beyond them.
    const int wj = GROUPED ? idx - 16 + lane : idx;
    const bool in_list = wj >= 0 && wj < quota;
    const uint32_t wyx = in_list ? kyx[wj] : 0u;
    const uint64_t wkey = in_list ? kkey[wj] : 0ull;
    // The frame's first slot publishes its keypoint count.
    if (slot == frame * n_features) {
        const int total = __reduce_add_sync(0xFFFFFFFFu, kept_l);
        // A detect-stage wait that expired leaves partial results: report it instead.
        if (lane == 0) call->counts[frame] = *call->status ? OF_ERR_TIMEOUT : total;
    }
    if (idx >= quota || idx >= kept) return;
    const int base = __reduce_add_sync(0xFFFFFFFFu, lane < level ? kept_l : 0);

    const uint32_t yx = GROUPED ? __shfl_sync(0xFFFFFFFFu, wyx, 16) : wyx;
    const uint64_t okey = GROUPED ? __shfl_sync(0xFFFFFFFFu, wkey, 16) : wkey;
    const int x = (int)(yx & 0xFFFFu), y = (int)(yx >> 16);
    // The patch, columns x - H .. x + H of rows y - H .. y + H, as aligned words
    // (images and pitches are multiples of 16 bytes; H <= border keeps its pixels
    // inside, and a word that would pass the caller's frame is read bytewise).
    uint32_t* const P = patch[threadIdx.x >> 5];
    const PatchWords pw = patch_words(x, y, H, width, height, OP_WORDS);
    const int sh = pw.sh;
    int rank = idx;
    {
        const uint8_t* const q = img + (size_t)(y - H) * pitch + (x - H - sh);
        uint32_t v[OP_WORDS];
#pragma unroll
        for (int k = 0; k < OP_WORDS; ++k) {
            const int i = lane + 32 * k, r = i / OP_WORDS, c = i - r * OP_WORDS;
            v[k] = i < pw.whole && c < pw.nw ? reinterpret_cast<const uint32_t*>(q + (size_t)r * pitch)[c] : 0u;
        }
        if (GROUPED) {
            // The run of this code in a window of 32 entries, and the better ones of it.
            const uint32_t mine = key_code(okey);
            auto count = [&](bool in, uint64_t k, uint32_t yx_k, uint32_t& run) {
                const bool same = in && key_code(k) == mine;
                run = __ballot_sync(0xFFFFFFFFu, same);
                return __popc(__ballot_sync(0xFFFFFFFFu, same && rank_less(okey, ~yx, k, ~yx_k)));
            };
            uint32_t run;
            int better = count(wj >= 0 && wj < kept, wkey, wyx, run);
            const bool more = (run >> 31) != 0u;
            int start = idx - 16 + __ffs((int)run) - 1;
            // The run beyond the window: four more windows at a time to one side.
            auto extend = [&](int w, int dir) {
                uint64_t k[4];
                uint32_t p[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = w + dir * 32 * j + lane;
                    k[j] = i >= 0 && i < kept ? kkey[i] : 0ull;
                    p[j] = i >= 0 && i < kept ? kyx[i] : 0u;
                }
                bool on = true;  // the run reaches the next window
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (on) {
                        const int at = w + dir * 32 * j;
                        better += count(at + lane >= 0 && at + lane < kept, k[j], p[j], run);
                        if (dir < 0 && run) start = at + __ffs((int)run) - 1;
                        on = dir < 0 ? (run & 1u) != 0u : (run >> 31) != 0u;
                    }
                return on;
            };
            if (run & 1u)
                for (int w = idx - 48; w > -32 && extend(w, -1); w -= 128) {}
            if (more)
                for (int w = idx + 16; w < kept && extend(w, 1); w += 128) {}
            rank = start + better;
        }
#pragma unroll
        for (int k = 0; k < OP_WORDS; ++k)
            if (lane + 32 * k < OP_SIZE) P[lane + 32 * k] = v[k];
        if (pw.tail && lane == (pw.whole & 31)) {
            const int x0 = x - H - sh + 4 * (pw.nw - 1);  // its first column, inside the frame
            const uint8_t* const last = img + (size_t)(y + H) * pitch + x0;
            uint32_t t = 0u;
            for (int i = 0; i < 4 && x0 + i < width; ++i) t |= (uint32_t)last[i] << (8 * i);
            P[pw.whole] = t;
        }
    }
    const int sc = lane == 0 ? (int)score[(size_t)y * spitch + x] : 0;
    // No tables: a level-0 image (scale^0 = 1; the allocation-free entry point).
    const float kx = fx ? fx[x] : (float)x, ky = fx ? fy[y] : (float)y;
    __syncwarp();

    // Lane = column u = lane - 15 (lanes beyond H repeat a column of the patch).
    const int u = lane - 15;
    const uint8_t* const col = reinterpret_cast<const uint8_t*>(P) + sh + H + min(max(u, -H), H);
    constexpr int RB = 4 * OP_WORDS;  // bytes per patch row
    int m10 = 0, m01 = 0;
    {
        // Rows of the disc in this column: |v| <= hv (none beyond the radius).
        const int hv = u >= -R && u <= R ? (int)sqrtf((float)(R * R - u * u)) : -1;
        const uint8_t* const mid = col + H * RB;
        int s0 = hv >= 0 ? mid[0] : 0;
#pragma unroll
        for (int v = 1; v <= 15; ++v) {
            const int up = v <= hv ? mid[-v * RB] : 0, dn = v <= hv ? mid[v * RB] : 0;
            s0 += up + dn;
            m01 += v * (dn - up);
        }
        m10 = u * s0;
    }
    m10 = __reduce_add_sync(0xFFFFFFFFu, m10);
    m01 = __reduce_add_sync(0xFFFFFFFFu, m01);

    // Harris sums over the 7 x 7 window: per row the lane's vertical smoothing
    // s = p(-1) + 2 p + p(+1) and difference d = p(+1) - p(-1), packed, meet the
    // neighbouring columns': gx = s(u+1) - s(u-1), gy = d(u-1) + 2 d(u) + d(u+1).
    int a = 0, b = 0, c = 0;
    {
        int pm = col[(H - 4) * RB], pc = col[(H - 3) * RB];
#pragma unroll
        for (int v = -3; v <= 3; ++v) {
            const int pn = col[(H + v + 1) * RB];
            const int sv = pm + 2 * pc + pn, dv = pn - pm;
            const uint32_t w = ((uint32_t)sv << 16) | (uint32_t)(dv + 512);
            const uint32_t wl = __shfl_up_sync(0xFFFFFFFFu, w, 1), wr = __shfl_down_sync(0xFFFFFFFFu, w, 1);
            const int gx = (int)(wr >> 16) - (int)(wl >> 16);
            const int gy = (int)(wl & 0xFFFFu) + (int)(wr & 0xFFFFu) + 2 * dv - 1024;
            a += gx * gx;
            b += gy * gy;
            c += gx * gy;
            pm = pc;
            pc = pn;
        }
    }
    const bool in = u >= -3 && u <= 3;
    a = __reduce_add_sync(0xFFFFFFFFu, in ? a : 0);
    b = __reduce_add_sync(0xFFFFFFFFu, in ? b : 0);
    c = __reduce_add_sync(0xFFFFFFFFu, in ? c : 0);

    if (lane == 0) {
        const int64_t key = (int64_t)(okey ^ 0x8000000000000000ull);
        // response = key / kden * (1/(4*7*255))^4 in float: key as hi * 2^32 + lo
        // (two 32-bit conversions), times the host-rounded scale -- no float64 here
        // (the FP64 pipe was the orientation kernel's busiest unit).
        const float keyf = fmaf((float)(int32_t)(key >> 32), 4294967296.0f, (float)(uint32_t)key);
        of_keypoint k;
        k.x = kx;
        k.y = ky;
        k.x_l = x;
        k.y_l = y;
        k.level = level;
        k.fast_score = sc + (call->t_lo - 1);  // the map holds s - (t_lo - 1)
        k.response = keyf * call->resp_scale;
        k.angle = (m10 == 0 && m01 == 0) ? 0.0f : atan2f((float)m01, (float)m10);
        k.A = a;
        k.B = b;
        k.C = c;
        k.m10 = m10;
        k.m01 = m01;
        k.reserved = 0;
        k.key = key;
        const size_t at = (size_t)frame * n_features + base + rank;
        const uint4* src = reinterpret_cast<const uint4*>(&k);
        uint4* d4 = reinterpret_cast<uint4*>(call->out + at);
#pragma unroll
        for (int i = 0; i < 4; ++i) d4[i] = src[i];
        if (call->host_out) {  // of_detect_host: the record into pinned host memory too
            uint4* h4 = reinterpret_cast<uint4*>(call->host_out + at);
#pragma unroll
            for (int i = 0; i < 4; ++i) h4[i] = src[i];
        }
    }
}

void launch_orient_range(const Img* imgs, int img_begin, int n_img, int slot_begin, int slot_end, const Call* call,
                         bool grouped, bool sparse, void* stream, const uint16_t* slot_img, bool pdl) {
    if (slot_end <= slot_begin || n_img <= 0) return;
    const int blocks = (slot_end - slot_begin + ORIENT_WARPS - 1) / ORIENT_WARPS;
    const auto kernel = grouped ? (sparse ? k_orient<true, true> : k_orient<true, false>)
                                : (sparse ? k_orient<false, true> : k_orient<false, false>);
    launch_chain(kernel, blocks, ORIENT_WARPS * 32, 0, (cudaStream_t)stream, pdl, 1, imgs, img_begin, n_img, slot_begin,
                 slot_end, call, slot_img);
}

void launch_orient(const Img* imgs, int n_img, const Call* call, int total_slots, bool grouped, bool sparse, void* stream,
                   bool pdl) {
    launch_orient_range(imgs, 0, n_img, 0, total_slots, call, grouped, sparse, stream, nullptr, pdl);
}

// ---------------------------------------------------------------- inspect
__global__ void k_inspect_cells(const Img* imgs, int img, int t_hi, int t_lo, uint8_t* dst) {
    const Img& I = imgs[img];
    const int n = I.ncx * I.ncy;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = (uint8_t)((t_hi != t_lo && I.cell[i]) ? t_hi : t_lo);
}

__global__ void k_inspect_cands(const Img* imgs, int img, int n, uint8_t* dst) {
    const Img& I = imgs[img];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int64_t* d = reinterpret_cast<int64_t*>(dst + 16 * (size_t)i);
        int32_t* d32 = reinterpret_cast<int32_t*>(dst + 16 * (size_t)i + 8);
        d[0] = (int64_t)(I.ckey[i] ^ 0x8000000000000000ull);
        d32[0] = (int32_t)(I.cyx[i] & 0xFFFFu);
        d32[1] = (int32_t)(I.cyx[i] >> 16);
    }
}

void launch_inspect_cells(const Img* imgs, int img, int t_hi, int t_lo, uint8_t* dst,
                          void* stream) {
    k_inspect_cells<<<64, 256, 0, (cudaStream_t)stream>>>(imgs, img, t_hi, t_lo, dst);
}

// S(p) from a dense copy of a map: 0 outside proposed tiles and below t_hi in
// flagged cells, else the offset score + t_lo - 1 (idempotent on final maps).
__global__ void k_inspect_score_final(const Img* imgs, int img, uint8_t* d, int w, int h, int t_hi, int t_lo,
                                      int border, int cell) {
    const Img& I = imgs[img];
    const int rw = w - 2 * border, rh = h - 2 * border;
    if (rw <= 0 || rh <= 0) return;
    const int64_t n = (int64_t)rw * rh;
    const int th = t_hi - t_lo + 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int x = border + (int)(i % rw), y = border + (int)(i / rw);
        uint8_t* p = d + (size_t)y * w + x;
        int v = *p;
        if (v == 0) continue;
        if (t_hi != t_lo && v < th && I.cell[(size_t)((y - border) / cell) * I.ncx + (x - border) / cell]) v = 0;
        if (I.pmask && I.pmask[(size_t)((y - border) >> 5) * 4 * I.tiles_x + ((x - I.tile_x0) >> 5)] == 0) v = 0;
        *p = (uint8_t)(v ? v + t_lo - 1 : 0);
    }
}

void launch_inspect_score_final(const Img* imgs, int img, uint8_t* d, int w, int h, int t_hi, int t_lo, int border,
                                int cell, void* stream) {
    k_inspect_score_final<<<256, 256, 0, (cudaStream_t)stream>>>(imgs, img, d, w, h, t_hi, t_lo, border, cell);
}

void launch_inspect_cands(const Img* imgs, int img, int n, uint8_t* dst, void* stream) {
    if (n <= 0) return;
    k_inspect_cands<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(imgs, img, n, dst);
}

}  // namespace ofk
