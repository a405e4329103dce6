// Pyramid resize: level l is a bilinear resize of level l-1 (the pyramid of
// an ORB front end, Sec. 1; level sizes "decrease exponentially", Sec. 6.1).
//
// Staged kernel (scales the fused kernel below does not take, or by choice):
// one launch resizes level l of every frame in the batch.  Each block owns a
// 128 x TH output tile (TH = 32 or 64, chosen by the autotuner): it stages the tile's source window in shared memory
// with aligned 16-byte loads (direct loads when the window is larger than the
// buffer, i.e. scales above ~2), then each thread writes 4 consecutive output
// pixels of TH/16 rows, one 32-bit store per row, with its 4 column weights kept
// in registers.  Source coordinates come from per-axis tables computed on
// the host: (i0 << 12) | a, a in [0, 2048] the weight of sample i0 + 1 in
// units of 1/2048; one rounding at the end:
//   out = ((2048-ay)((2048-ax)p00 + ax p01) + ay((2048-ax)p10 + ax p11) + 2^21) >> 22.
// Exact int32 arithmetic: the largest intermediate is 2048*2048*255 < 2^31.
#include <cuda_runtime.h>

#include "of_internal.h"
#include "of_launch.cuh"
#include "of_tma.cuh"

namespace ofk {

__device__ __forceinline__ int find_job(const int32_t* __restrict__ prefix, int n, int b) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Shared-memory source window: up to RS_SW x RS_SH bytes (enough for scales
// up to 2 with a 128 x 64 output tile).
constexpr int RS_SW = 288;
constexpr int RS_SH = 136;

__device__ __forceinline__ int bilerp(int p00, int p01, int p10, int p11, int ax, int ay) {
    const int top = (2048 - ax) * p00 + ax * p01;
    const int bot = (2048 - ax) * p10 + ax * p11;
    return ((2048 - ay) * top + ay * bot + (1 << 21)) >> 22;
}

template <int TH>
__global__ void __launch_bounds__(RS_THREADS)
k_resize(const Resize* __restrict__ jobs, const int32_t* __restrict__ prefix, int n_jobs) {
    constexpr int RS_RPT = TH / (RS_THREADS / 32);  // output rows per thread
    __shared__ __align__(16) uint8_t win[RS_SH * RS_SW];
    __shared__ int32_t yt[TH];
    __shared__ int32_t sjob, sx0s, sy0s, sbytes, srows;
    const int b = blockIdx.x;
    if (threadIdx.x == 0) sjob = find_job(prefix, n_jobs, b);
    __syncthreads();
    const int j = sjob;
    const Resize& J = jobs[j];
    const int t = b - __ldg(prefix + j);
    const int tx = t % J.tiles_x, ty = t / J.tiles_x;
    const int X0 = tx * RS_TILE_W, Y0 = ty * TH;
    const int nx = min(RS_TILE_W, J.dw - X0), ny = min(TH, J.dh - Y0);
    const int sw = J.sw, sh = J.sh;
    for (int i = threadIdx.x; i < TH; i += blockDim.x) yt[i] = i < ny ? __ldg(J.ytab + Y0 + i) : 0;
    if (threadIdx.x == 0) {
        // Source window of the tile: columns [sx0, sx1], rows [sy0, sy1].
        const int sx0 = (__ldg(J.xtab + X0) >> 12) & ~15;
        const int sx1 = min((__ldg(J.xtab + X0 + nx - 1) >> 12) + 1, sw - 1);
        const int sy0 = __ldg(J.ytab + Y0) >> 12;
        const int sy1 = min((__ldg(J.ytab + Y0 + ny - 1) >> 12) + 1, sh - 1);
        sx0s = sx0;
        sy0s = sy0;
        sbytes = ((sx1 - sx0) / 16 + 1) * 16;
        srows = sy1 - sy0 + 1;
    }
    __syncthreads();
    const int sx0 = sx0s, sy0 = sy0s, wbytes = sbytes, wrows = srows;
    const bool staged = wbytes <= RS_SW && wrows <= RS_SH;  // uniform per block
    if (staged) {
        const int cpr = wbytes / 16;
        for (int i = threadIdx.x; i < wrows * cpr; i += blockDim.x) {
            const int r = i / cpr, k = i - r * cpr;
            const int ix = sx0 + 16 * k;
            const uint8_t* p = J.src + (size_t)(sy0 + r) * J.spitch + ix;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (ix + 16 <= sw) {
                v = __ldg(reinterpret_cast<const uint4*>(p));  // src and spitch are 16-byte aligned
            } else {
                // Ragged end of the row: bytewise, in bounds.
                uint32_t w0 = 0u, w1 = 0u, w2 = 0u, w3 = 0u;
                for (int q = 0; q < 16 && ix + q < sw; ++q) {
                    const uint32_t byte = (uint32_t)__ldg(p + q) << (8 * (q & 3));
                    if (q < 4) w0 |= byte; else if (q < 8) w1 |= byte; else if (q < 12) w2 |= byte; else w3 |= byte;
                }
                v = make_uint4(w0, w1, w2, w3);
            }
            *reinterpret_cast<uint4*>(win + r * RS_SW + 16 * k) = v;
        }
    }
    __syncthreads();

    // Each thread: 4 consecutive columns, rows ly, ly + 16, ...
    const int lx = (threadIdx.x & 31) * 4, ly0 = threadIdx.x >> 5;
    if (lx >= nx) return;
    const int n = min(4, nx - lx);
    int x0[4], x1[4], ax[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = i < n ? __ldg(J.xtab + X0 + lx + i) : __ldg(J.xtab + X0 + lx);
        x0[i] = e >> 12;
        ax[i] = e & 4095;
        x1[i] = min(x0[i] + 1, sw - 1);
    }
#pragma unroll
    for (int rr = 0; rr < RS_RPT; ++rr) {
        const int ly = ly0 + rr * (RS_THREADS / 32);
        if (ly >= ny) break;
        const int y0 = yt[ly] >> 12, ay = yt[ly] & 4095;
        const int y1 = min(y0 + 1, sh - 1);
        uint32_t packed = 0;
        if (staged) {
            const uint8_t* r0 = win + (y0 - sy0) * RS_SW - sx0;
            const uint8_t* r1 = win + (y1 - sy0) * RS_SW - sx0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                packed |= (uint32_t)bilerp(r0[x0[i]], r0[x1[i]], r1[x0[i]], r1[x1[i]], ax[i], ay) << (8 * i);
        } else {
            const uint8_t* r0 = J.src + (size_t)y0 * J.spitch;
            const uint8_t* r1 = J.src + (size_t)y1 * J.spitch;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                packed |= (uint32_t)bilerp(__ldg(r0 + x0[i]), __ldg(r0 + x1[i]), __ldg(r1 + x0[i]),
                                           __ldg(r1 + x1[i]), ax[i], ay)
                          << (8 * i);
        }
        uint8_t* d = J.dst + (size_t)(Y0 + ly) * J.dpitch + X0 + lx;
        if (n == 4) {
            *reinterpret_cast<uint32_t*>(d) = packed;  // X0 + lx is a multiple of 4, dpitch of 16
        } else {
            for (int i = 0; i < n; ++i) d[i] = (uint8_t)(packed >> (8 * i));
        }
    }
}

void launch_resize(const Resize* jobs, const int32_t* tile_prefix, int n_jobs, int n_tiles, int tile_h,
                   void* stream) {
    if (n_tiles <= 0) return;
    if (tile_h == 32)
        k_resize<32><<<n_tiles, RS_THREADS, 0, (cudaStream_t)stream>>>(jobs, tile_prefix, n_jobs);
    else
        k_resize<64><<<n_tiles, RS_THREADS, 0, (cudaStream_t)stream>>>(jobs, tile_prefix, n_jobs);
}

// ---------------------------------------------------------------------------
// Fused pyramid: a run of levels in one launch, no level waits for another.
//
// Every level is resized from the one before it, so level by level the pyramid
// is a chain of dependent launches (7 for 8 levels: 38 us for one 1080p frame,
// nearly all of it latency), each reading back what the last one wrote.  Here a
// block owns a rectangle of every level of the run -- equal shares of the
// image -- and computes it from its piece of the source level alone: it loads
// that piece once (one TMA box), then resizes it level by level in shared
// memory, each level over its own rectangle plus the few pixels its rectangles
// of the later levels need (7 levels at scale 1.2: 1.3 times the pixels for a
// 128 x 128 source piece), and writes what it owns to global memory.  Pixels
// near the seams are computed by two blocks, identically.
//
// The bilinear value factors into a horizontal and a vertical step, both exact
// in unsigned 32-bit arithmetic when every weight is doubled:
//   h(r, x) = (4096 - 2ax) S[r][x0] + 2ax S[r][x0 + 1]           (< 2^20)
//   v       = (4096 - 2ay) h(y0, x) + 2ay h(y0 + 1, x) + 2^23    (< 2^32)
//   out     = v >> 24 = ((sum of the original products) + 2^21) >> 22.
// h is one __dp2a_lo or __dp2a_hi (two 16 x 8-bit products) on a byte pair;
// one __byte_perm picks the byte pairs of two outputs into the low and high
// halves of a word; out is byte 3 of v, so four outputs pack with three byte
// permutes.  Where a source index is clamped (x0 = w - 1, y0 = h - 1) the
// tables give that sample's partner weight 0, so what lies past the edge never
// contributes.  The plan's tables (pyramid_axis) hold, per tile column and row,
// every level's ranges, byte selectors, weights and source rows, relative to
// the tile.  A thread owns 4 columns of a strip of rows and keeps the
// horizontal values of the two source rows under the current output row in
// registers as it moves down.  Measured (stage time): one 1080p frame 38 -> 16
// us, one 4K frame 51 -> 28, 64 frames of four sizes 166 -> 122, 128 1080p
// frames 459 -> 340; batches are bound by instruction issue (72 %).

// Horizontal pass of one source row for a thread's 4 columns.
__device__ __forceinline__ void hrow(const uint32_t* __restrict__ row, uint32_t wa, uint32_t wb, uint32_t sel,
                                     const uint32_t (&wgt)[4], uint32_t (&h)[4]) {
    const uint32_t a0 = row[wa], a1 = row[wa + 1], b0 = row[wb], b1 = row[wb + 1];
    const uint32_t p01 = __byte_perm(a0, a1, sel), p23 = __byte_perm(b0, b1, sel >> 16);
    h[0] = __dp2a_lo(wgt[0], p01, 0u);
    h[1] = __dp2a_hi(wgt[1], p01, 0u);
    h[2] = __dp2a_lo(wgt[2], p23, 0u);
    h[3] = __dp2a_hi(wgt[3], p23, 0u);
}

__global__ void __launch_bounds__(PY_THREADS, 4)
k_pyramid(const PyrJob* __restrict__ jobs, const uint2* __restrict__ items, const CUtensorMap* __restrict__ maps,
          const Call* __restrict__ call, int s_bytes, int t_bytes, int x_words) {
    // The piece of the source level (and of levels 2, 4, ...), of levels 1, 3, ..., then the tables.
    extern __shared__ __align__(128) uint8_t pdyn[];
    __shared__ __align__(8) uint64_t mbar;
    uint8_t* const S = pdyn + ((128u - (smem_u32(pdyn) & 127u)) & 127u);
    uint8_t* const T = S + s_bytes;
    int32_t* const xs = reinterpret_cast<int32_t*>(T + t_bytes);
    int32_t* const ys = xs + x_words;
    const int tid = threadIdx.x;
    pdl_trigger();
    const uint2 it = __ldg(items + blockIdx.x);  // (job, (tile row << 16) | tile column)
    const PyrJob& J = jobs[it.x];
    const int32_t* const xg = J.xblk + (size_t)(it.y & 0xFFFFu) * J.xstride;
    const int32_t* const yg = J.yblk + (size_t)(it.y >> 16) * J.ystride;
    if (tid == 0) {
        mbar_init(&mbar, 1);
        fence_barrier_init();
        tensormap_acquire(maps + it.x);
        pdl_wait();  // a later run reads the levels of the run before it
        mbar_arrive_expect_tx(&mbar, (uint32_t)(J.box_w * J.box_h));
        tma_load_2d(S, maps + it.x, __ldg(xg), __ldg(yg), &mbar);
    }
    for (int i = tid; i < J.xstride / 4; i += PY_THREADS)
        reinterpret_cast<int4*>(xs)[i] = __ldg(reinterpret_cast<const int4*>(xg) + i);
    for (int i = tid; i < J.ystride / 4; i += PY_THREADS)
        reinterpret_cast<int4*>(ys)[i] = __ldg(reinterpret_cast<const int4*>(yg) + i);
    const int nl = J.nl;
    __syncthreads();
    pdl_wait();
    const bool ok = mbar_wait(&mbar, 0);
    if (__syncthreads_or(!ok)) {
        if (tid == 0) {
            atomicOr(call->status, OF_DEV_TIMEOUT);
            mbar_wait(&mbar, 0, OF_WAIT_LIMIT_NS / 8);  // let the copy land before the shared memory goes away
        }
        return;
    }
    const int32_t* xe = xs + 4 * (nl + 1);
    const int32_t* ye = ys + 4 * (nl + 1);
    int spw = J.box_w / 4;  // words per row of the level being read
    for (int l = 1; l <= nl; ++l) {
        const int4 hx = reinterpret_cast<const int4*>(xs)[l], hy = reinterpret_cast<const int4*>(ys)[l];
        const uint32_t* const src = reinterpret_cast<const uint32_t*>((l & 1) ? S : T);
        uint32_t* const dst = reinterpret_cast<uint32_t*>((l & 1) ? T : S);
        const int ncg = hx.y & 255, nr = hy.y & 0xFFFF, dpw = hy.y >> 16;
        const uint32_t m = (uint32_t)hx.y >> 8;
        // Strips of rp rows: as many as the threads give (strip = tid / ncg).
        const int strips = (int)(m >> 8), strip = (int)(((uint32_t)tid * m) >> 16), cg = tid - strip * ncg;
        if (ncg > 0 && strip < strips) {
            const int rp = (int)(((float)(nr + strips - 1) + 0.5f) * __frcp_rn((float)strips));  // ceil(nr / strips)
            int r = strip * rp;
            const int re = min(r + rp, nr);
            const int4 ea = *reinterpret_cast<const int4*>(xe + 8 * cg);
            const int2 eb = *reinterpret_cast<const int2*>(xe + 8 * cg + 4);
            const uint32_t wa = (uint32_t)ea.x & 0xFFFFu, wb = (uint32_t)ea.x >> 16, sel = (uint32_t)ea.y;
            const uint32_t wgt[4] = {(uint32_t)ea.z, (uint32_t)ea.w, (uint32_t)eb.x, (uint32_t)eb.y};
            const int x = hx.x + 4 * cg;
            // Owned rows of the strip: none when the columns are another tile's.
            const bool mine = x >= hx.z && x < hx.w;
            const int o0 = mine ? hy.z - hy.x : nr, o1 = hy.w - hy.x;
            const int pitch = J.dpitch[l - 1];
            // Word stores: x and the pitch are multiples of 4; a level's rows are padded to 16 bytes.
            uint8_t* g = J.dst[l - 1] + (ptrdiff_t)(hy.x + r) * pitch + x;
            uint32_t* d = dst + r * dpw + cg;
            const bool keep = l < nl;
            uint32_t ha[4], hb[4] = {0u, 0u, 0u, 0u};
            int next = -1;  // word offset of the row below the last one read
#pragma unroll 2
            for (; r < re; ++r, g += pitch, d += dpw) {
                const uint32_t e = (uint32_t)ye[r];
                const int off = (int)(e >> 16);
                const uint32_t a2 = e & 0xFFFFu;
                // Consecutive output rows mostly read consecutive source rows: the
                // upper one is then the last lower one.  Only the other lanes branch.
#pragma unroll
                for (int i = 0; i < 4; ++i) ha[i] = hb[i];
                if (off != next) hrow(src + off, wa, wb, sel, wgt, ha);
                next = off + spw;
                hrow(src + next, wa, wb, sel, wgt, hb);
                uint32_t v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = (4096u - a2) * ha[i] + a2 * hb[i] + (1u << 23);
                const uint32_t packed =
                    __byte_perm(__byte_perm(v[0], v[1], 0x0073), __byte_perm(v[2], v[3], 0x0073), 0x5410);
                if (keep) *d = packed;
                if (r >= o0 && r < o1) *reinterpret_cast<uint32_t*>(g) = packed;
            }
        }
        xe += 8 * ncg;
        ye += nr;
        spw = dpw;
        __syncthreads();
    }
}

int pyramid_smem(int s_bytes, int t_bytes, int x_words, int y_words) {
    return s_bytes + t_bytes + 4 * (x_words + y_words) + 128;
}

void launch_pyramid(const PyrJob* jobs, const uint2* items, int n_tiles, const CUtensorMap* maps, const Call* call,
                    int s_bytes, int t_bytes, int x_words, int y_words, void* stream, bool pdl) {
    if (n_tiles <= 0) return;
    launch_chain(k_pyramid, n_tiles, PY_THREADS, pyramid_smem(s_bytes, t_bytes, x_words, y_words),
                 (cudaStream_t)stream, pdl, 1, jobs, items, maps, call, s_bytes, t_bytes, x_words);
}

// Raised once to the largest size any plan may use, so graphs captured for
// different plans never depend on which plan set it last.
bool pyramid_raise_smem() {
    return cudaFuncSetAttribute(k_pyramid, cudaFuncAttributeMaxDynamicSharedMemorySize, PY_MAX_SMEM) == cudaSuccess;
}

}  // namespace ofk
