// Tile-proposal network: forward, backward, Adam, checkpoints.
//
// The paper has no learned part; this network decides, per 32 x 32 tile of a
// pyramid level, whether the exact detector needs to run there.  Input: the
// tile with a 16-pixel halo (64 x 64 uint8, zero outside the image),
// normalised to (v - 128) / 64.  Layers (3 x 3 kernels, stride 2, padding 1,
// ReLU): 1 -> 8 channels (32 x 32), 8 -> 16 (16 x 16), 16 -> 16 (8 x 8);
// global average pool; linear 16 -> 1 logit.  Weights are stored and used as
// bf16 (rounded from fp32 master copies that Adam updates); every product is
// accumulated in fp32.  One block per tile; activations stay in shared memory;
// inference and training run on the tensor cores.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "of_edge.cuh"
#include "of_internal.h"
#include "ofast.h"

namespace ofk {
void set_last_error(const std::string& msg);
}

namespace tn {

constexpr int S0 = 64, S2 = 16, S3 = 8;  // spatial sizes (64, 32, 16, 8)
constexpr int C1 = 8, C2 = 16, C3 = 16;
// Flat parameter layout.
constexpr int W1 = 0, B1 = W1 + C1 * 9, W2 = B1 + C1, B2 = W2 + C2 * C1 * 9, W3 = B2 + C2,
              B3 = W3 + C3 * C2 * 9, WF = B3 + C3, BF = WF + C3, NP = BF + 1;
static_assert(NP == 3585, "parameter count");
// Behind the gradient, on 8 bytes: the loss and the last bias' gradient, sums over all patches of numbers of
// both signs, as doubles (the latter rounded where it is read).
constexpr int LOSS_AT = (NP + 1) / 2 * 2, GRAD_WORDS = LOSS_AT + 4;

}  // namespace tn

struct of_tcnn {
    float* master = nullptr;  // fp32 master weights [NP]
    __nv_bfloat16* w = nullptr;  // bf16 compute weights [NP]
    float* grad = nullptr;    // fp32 gradients [NP] (the last bias' apart), then (LOSS_AT) what a step sums in double
    float* m = nullptr;       // Adam moments
    float* v = nullptr;
    int64_t step = 0;
    int device = 0;
};

namespace tn {

__device__ __forceinline__ float relu(float x) { return x > 0.f ? x : 0.f; }

// Source of the 64 x 64 input patches: a dense tile array, or the proposal
// tiles of pyramid levels read in place.  Proposal tile t is quarter t & 3 of
// detect tile t / 4 of the plan's item table ((image, (y0 << 16) | x0): the
// 128 x 32 tiles of all images in order), so no search over the images.
struct PatchSrc {
    const uint8_t* tiles;   // dense: n x 4096 bytes, or nullptr
    const ofk::Img* imgs;   // in place: image descriptors
    const uint2* items;     // in place: the detect tiles
};

// A 64 x 64 patch is 256 16-byte chunks (4 per row).  Chunk q of tile t; pixels
// outside the image are 0.  Level images and their pitches are multiples of
// 16 bytes, and a patch starts at a multiple of 16, so a chunk is one aligned
// load (whole inside the row's pitch; bytewise where it would pass the end of a
// caller's frame); bytes past the row's w are cleared.
struct Patch {
    const uint8_t* p;       // dense: the tile; in place: the level image
    int x0, y0, w, h, pitch;  // in place; pitch 0: dense
};

__device__ __forceinline__ Patch find_patch(const PatchSrc& S, int t) {
    Patch P;
    if (S.tiles) {
        P.p = S.tiles + (size_t)t * S0 * S0;
        P.x0 = P.y0 = P.w = P.h = P.pitch = 0;
        return P;
    }
    const uint2 e = __ldg(S.items + (t >> 2));
    const ofk::Img& I = S.imgs[e.x];
    P.p = I.img;
    P.x0 = (int)(e.y & 0xFFFFu) + 32 * (t & 3) - 16;
    P.y0 = (int)(e.y >> 16) - 16;
    P.w = I.w;
    P.h = I.h;
    P.pitch = I.pitch;
    return P;
}

__device__ __forceinline__ uint4 load_chunk(const Patch& P, int q) {
    if (P.pitch == 0) {
        const uint8_t* p = P.p + 16 * q;
        if ((reinterpret_cast<uintptr_t>(P.p) & 15) == 0) return __ldg(reinterpret_cast<const uint4*>(p));
        uint32_t v[4] = {0u, 0u, 0u, 0u};  // a caller's unaligned tile array
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i >> 2] |= (uint32_t)__ldg(p + i) << (8 * (i & 3));
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
    const int x = P.x0 + 16 * (q & 3), y = P.y0 + (q >> 2);
    if (x < 0 || x >= P.w || y < 0 || y >= P.h) return make_uint4(0u, 0u, 0u, 0u);
    const uint8_t* const p = P.p + (size_t)y * P.pitch + x;
    const int n = ofk::chunk_bytes(x, P.w);
    if (!ofk::chunk_whole(n, y, P.h)) {  // at most 15 bytes
        uint32_t v[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < 15; ++i)
            if (i < n) v[i >> 2] |= (uint32_t)__ldg(p + i) << (8 * (i & 3));
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
    uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
    if (n < 16) {
        uint32_t* m = &v.x;
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] &= n >= 4 * i + 4 ? 0xFFFFFFFFu : n <= 4 * i ? 0u : (1u << (8 * (n - 4 * i))) - 1u;
    }
    return v;
}

// ---------------------------------------------------------------------------
// Inference on the tensor cores, without losing precision.
//
// An fp32 activation is the exact sum of three bf16 numbers (its leading 8
// significant bits, the next 8, the last 8: truncations), the weights are bf16
// already, so every product of a layer is an exact bf16 product and the layer
// is a matrix product with three times the depth.  The tensor cores' fp32
// accumulation truncates, though: a long chain of the leading parts would bias
// the logits (5e-7 of their norm).  So the leading parts' products of one
// 16-deep step are summed from zero and added to the running sum with an fp32
// addition; only the lower parts, 2^-8 and 2^-16 of the size, stay in a chain.
// Against 64 bits the logits are 7.2e-8 of their norm off (median of 48 batches,
// committed network), the fp32 FMA kernel's were 8.7e-8.
//
// The layers are far too narrow (8 or 16 channels) for tcgen05's 128-row
// tiles to be filled by channels, and a sum from zero per step would cost a
// TMEM read per step, so warp-level m16n8k16 products with pixels as rows and
// channels as columns carry the work; all weight fragments stay in registers.
// Activations are stored channels-last, 8 channels = 16 bytes per pixel, one
// plane per part (and per channel half), columns split by parity, so that
// each tap of 8 neighbouring output pixels is 128 contiguous bytes: one 8 x 8
// matrix of ldmatrix, no im2col copy and no bank conflict.  The input (exact
// in bf16) keeps rows of pixels: an output's three taps of a row and a zero
// weight are two aligned words.
//
// A block of 8 warps takes one tile at a time, two blocks per SM; a layer's
// planes have buffers of their own, so a tile needs two barriers, and the next
// tile's pixels are staged while layer 2 runs.  Layer 3 is four products' rows
// of work: four warps do it, both channel halves from one read of the
// activations, while the other four start on the next tile's layer 1.  Bound by
// shared memory (~2430 wavefronts per tile, 61 % of its rate).  16,384 patches:
// 755 us as fp32 FMAs over shared-memory operands, 397 us register-blocked with
// packed fp32 FMAs (the smem reads of the weights then bound it), 240 us on the
// tensor cores with a channel half of layer 3 per warp (each reading all
// activations), 219 us here (219.6, 220.1 and 221.2 us with 4,
// 5 and 7 instead of 6 layer-1 products per warp that also does layer 3).
constexpr int FWD_THREADS = 256, FWD_BLOCKS = 2;
constexpr int TI_ROW = 48, TI_X = 4;                       // input rows: words per row (pixel pairs), word of pixel 0
constexpr int TI_BYTES = 65 * TI_ROW * 4;                  // row 0: zeros
constexpr int T1_ROW = 33, T1_O = 17;                      // layer-1 rows: 17 even padded columns, then 16 odd ones
constexpr int T1_PLANE = 33 * T1_ROW * 16;                 // one part: 33 rows (row 0: zeros), 8 channels
constexpr int T2_ROW = 21, T2_O = 13;                      // layer-2 rows: 9 even columns, (gap), 8 odd ones
constexpr int T2_PLANE = 17 * T2_ROW * 16;                 // one part and channel half: 17 rows
constexpr int FWD_RED = 2 * 4 * C3;                        // per tile parity and row pair: channel sums
constexpr int FWD_B3 = 18 * 32;                            // layer-3 weight fragments: a word pair per lane, tap and channel half
constexpr int FWD_SMEM = TI_BYTES + 3 * T1_PLANE + 6 * T2_PLANE + FWD_RED * 4 + FWD_B3 * 8;
constexpr int FWD_L1A = 6;                                 // layer-1 products of each of the four warps that also do layer 3
static_assert(TI_BYTES % 16 == 0 && T1_PLANE % 16 == 0 && T2_PLANE % 16 == 0, "16-byte rows for ldmatrix");

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(a)
                 : "memory");
}
// d = a b + c, a 16 x 16 (pixels x depth), b 16 x 8 (depth x channels).
__device__ __forceinline__ void mma16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2], const float (&c)[4]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %11, %12, %13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
__device__ __forceinline__ void mma8(float (&d)[4], const uint32_t (&a)[2], uint32_t b, const float (&c)[4]) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %8, %9, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(b), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// The three bf16 parts of two values (channels 2t, 2t + 1), packed:
// truncations, so that finite values never round up to infinity; an infinity
// is its own leading part.
__device__ __forceinline__ void split3(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
    auto rest = [](float v) {
        const float r = v - __uint_as_float(__float_as_uint(v) & 0xFFFF0000u);
        return r;
    };
    const bool xi = fabsf(x) > 3.402823466e38f, yi = fabsf(y) > 3.402823466e38f;
    const float rx = xi ? 0.f : rest(x), ry = yi ? 0.f : rest(y);
    const float sx = rest(rx), sy = rest(ry);
    h = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
    m = __byte_perm(__float_as_uint(rx), __float_as_uint(ry), 0x7632);
    l = __byte_perm(__float_as_uint(sx), __float_as_uint(sy), 0x7632);
}

// split3 into the planes of the three parts, `plane` bytes apart.
__device__ __forceinline__ void store3(uint8_t* d, int plane, float x, float y) {
    uint32_t h, m, l;
    split3(x, y, h, m, l);
    *reinterpret_cast<uint32_t*>(d) = h;
    *reinterpret_cast<uint32_t*>(d + plane) = m;
    *reinterpret_cast<uint32_t*>(d + 2 * plane) = l;
}

// Two consecutive input channels (or taps) of a weight matrix as one fragment word.
__device__ __forceinline__ uint32_t pack_w(const __nv_bfloat16* __restrict__ w, int i0, int i1) {
    const uint32_t lo = i0 >= 0 ? __bfloat16_as_ushort(w[i0]) : 0u, hi = i1 >= 0 ? __bfloat16_as_ushort(w[i1]) : 0u;
    return lo | (hi << 16);
}

// Chunk q (16 pixels) of the patch as bf16 (v - 128) / 64, exact, into the input plane.
__device__ __forceinline__ void stage_bf16(uint32_t* __restrict__ in, int q, const uint4& v) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t wd = u[i >> 1];
        const float a = fmaf(__uint_as_float(__byte_perm(wd, 0x4B000000u, (i & 1) ? 0x7552 : 0x7550)), 1.f / 64.f, -131074.f);
        const float b = fmaf(__uint_as_float(__byte_perm(wd, 0x4B000000u, (i & 1) ? 0x7553 : 0x7551)), 1.f / 64.f, -131074.f);
        o[i] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
    }
    uint4* d = reinterpret_cast<uint4*>(in + ((q >> 2) + 1) * TI_ROW + TI_X + 8 * (q & 3));
    d[0] = make_uint4(o[0], o[1], o[2], o[3]);
    d[1] = make_uint4(o[4], o[5], o[6], o[7]);
}

__global__ void __launch_bounds__(FWD_THREADS, FWD_BLOCKS)
k_forward_fast(PatchSrc src, int n, const __nv_bfloat16* __restrict__ wq, float* __restrict__ logits) {
    extern __shared__ __align__(128) uint8_t fsm[];
    uint32_t* const in = reinterpret_cast<uint32_t*>(fsm);
    uint8_t* const p1 = fsm + TI_BYTES;
    uint8_t* const p2 = p1 + 3 * T1_PLANE;
    float* const red = reinterpret_cast<float*>(p2 + 6 * T2_PLANE);
    uint2* const b3 = reinterpret_cast<uint2*>(red + FWD_RED);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    // Zero the planes once: the pad words are never written afterwards.
    for (int i = tid; i < (TI_BYTES + 3 * T1_PLANE + 6 * T2_PLANE) / 16; i += FWD_THREADS)
        reinterpret_cast<uint4*>(fsm)[i] = make_uint4(0u, 0u, 0u, 0u);

    // Weight fragments.  Layer 1: depth 4 ky + j, j = 0 a zero weight (the pixel
    // two to the left), j = kx + 1; layer 2: two taps of 8 channels per step, the
    // ninth alone; layer 3: a tap of 16 channels per step, in shared memory.
    uint32_t b1[2], b2[2][4][2], b2e[2];
    {
        auto w1 = [&](int k) {  // depth k of layer 1, channel g; -1: zero weight
            return k < 12 && (k & 3) ? W1 + g * 9 + (k >> 2) * 3 + (k & 3) - 1 : -1;
        };
        b1[0] = pack_w(wq, w1(2 * t4), w1(2 * t4 + 1));
        b1[1] = pack_w(wq, w1(2 * t4 + 8), w1(2 * t4 + 9));
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = W2 + (8 * j + g) * C1 * 9 + 2 * t4 * 9;  // output channel 8 j + g, input channel 2 t
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                b2[j][s][0] = pack_w(wq, r + 2 * s, r + 9 + 2 * s);
                b2[j][s][1] = pack_w(wq, r + 2 * s + 1, r + 9 + 2 * s + 1);
            }
            b2e[j] = pack_w(wq, r + 8, r + 9 + 8);
        }
        for (int i = warp; i < 18; i += FWD_THREADS / 32) {
            const int k = i >> 1, r = W3 + (8 * (i & 1) + g) * C2 * 9 + 2 * t4 * 9;
            b3[i * 32 + lane] = make_uint2(pack_w(wq, r + k, r + 9 + k), pack_w(wq, r + 8 * 9 + k, r + 9 * 9 + k));
        }
    }
    auto bias = [&](int i) { return __bfloat162float(wq[i]); };
    const float bb1[2] = {bias(B1 + 2 * t4), bias(B1 + 2 * t4 + 1)};
    const float bb2[4] = {bias(B2 + 2 * t4), bias(B2 + 2 * t4 + 1), bias(B2 + 8 + 2 * t4), bias(B2 + 9 + 2 * t4)};
    const float bb3[4] = {bias(B3 + 2 * t4), bias(B3 + 2 * t4 + 1), bias(B3 + 8 + 2 * t4), bias(B3 + 9 + 2 * t4)};
    const float wf = bias(WF + (lane & 15)), bf = bias(BF);
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};

    // ldmatrix row addresses of this lane (relative to the plane and the output row).
    auto col1 = [](int kx) { return kx == 1 ? T1_O : kx >> 1; };  // E[x], O[x], E[x + 1]
    uint32_t off2[4], off2e;
    {
        const int x = (lane & 7) + 8 * ((lane >> 3) & 1);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int tap = 2 * s + (lane >> 4);
            off2[s] = (uint32_t)(((tap / 3) * T1_ROW + col1(tap % 3) + x) * 16);
        }
        off2e = (uint32_t)((2 * T1_ROW + 1 + x) * 16);
    }
    const uint32_t s1 = smem_addr(p1), s2 = smem_addr(p2);
    // Layer 3, warps 0 to 3: output row 2 warp + (bit 3 of the lane), column lane & 7, channel half = bit 4.
    const uint32_t a3base =
        s2 + (uint32_t)((lane >> 4) * T2_PLANE + (2 * (2 * warp + ((lane >> 3) & 1)) * T2_ROW + (lane & 7)) * 16);

    auto finish = [&](int t, int par) {  // warp 0: the head of a finished tile
        const float* r = red + par * 4 * C3 + (lane & 15);
        float z = ((r[0] + r[C3]) + (r[2 * C3] + r[3 * C3])) * (1.f / 64.f) * wf;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
        if (lane == 0) logits[t] = z + bf;
    };

    int t = blockIdx.x, last = -1;
    __syncthreads();
    if (t < n) stage_bf16(in, tid, load_chunk(find_patch(src, t), tid));
    __syncthreads();
    for (int par = 0; t < n; par ^= 1) {
        const int tn = t + gridDim.x;
        uint4 pix = make_uint4(0u, 0u, 0u, 0u);
        if (tn < n) pix = load_chunk(find_patch(src, tn), tid);
        // Layer 1: 64 products of 16 pixels (a row's half: even columns 2 g + 16 h, odd ones).
        // Warps 4 to 7, without a part of layer 3, start earlier and take more of them.
        const int l1_0 = warp < 4 ? warp : 4 * FWD_L1A + warp - 4, l1_1 = warp < 4 ? 4 * FWD_L1A : 64;
#pragma unroll 2
        for (int i = l1_0; i < l1_1; i += 4) {
            const int y = i >> 1, h = i & 1;
            const uint32_t* r = in + (2 * y + (t4 >> 1)) * TI_ROW + TI_X - 1 + 2 * g + 16 * h + (t4 & 1);
            const uint32_t* r2 = in + (2 * y + 2) * TI_ROW + TI_X - 1 + 2 * g + 16 * h + t4;
            uint32_t a[4] = {r[0], r[1], 0u, 0u};
            if (t4 < 2) {
                a[2] = r2[0];
                a[3] = r2[1];
            }
            float d[4];
            mma16(d, a, b1, zero);
            uint8_t* o = p1 + ((y + 1) * T1_ROW + g + 8 * h) * 16 + 4 * t4;
            store3(o + T1_O * 16, T1_PLANE, relu(d[0] + bb1[0]), relu(d[1] + bb1[1]));  // even columns: odd padded ones
            store3(o + 16, T1_PLANE, relu(d[2] + bb1[0]), relu(d[3] + bb1[1]));
        }
        __syncthreads();
        if (warp == 0 && last >= 0) finish(last, par ^ 1);
        if (tn < n) stage_bf16(in, tid, pix);
        // Layer 2: two output rows per warp, 16 pixels x 16 channels each.
#pragma unroll 1
        for (int y = warp; y < S2; y += 8) {
            const uint32_t row = s1 + (uint32_t)(2 * y * T1_ROW * 16);
            float acc[2][4] = {}, low[2][4] = {};
#pragma unroll
            for (int s = 0; s < 5; ++s) {
                uint32_t ah[4], am[4], al[4];
                if (s < 4) {
                    ldsm4(ah, row + off2[s]);
                    ldsm4(am, row + off2[s] + T1_PLANE);
                    ldsm4(al, row + off2[s] + 2 * T1_PLANE);
                } else {
                    uint32_t q[2];
                    ldsm2(q, row + off2e);
                    ah[0] = q[0], ah[1] = q[1];
                    ldsm2(q, row + off2e + T1_PLANE);
                    am[0] = q[0], am[1] = q[1];
                    ldsm2(q, row + off2e + 2 * T1_PLANE);
                    al[0] = q[0], al[1] = q[1];
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float d[4];
                    if (s < 4) {
                        mma16(d, ah, b2[j][s], zero);
                        mma16(low[j], al, b2[j][s], low[j]);
                        mma16(low[j], am, b2[j][s], low[j]);
                    } else {
                        const uint32_t h2[2] = {ah[0], ah[1]}, m2[2] = {am[0], am[1]}, l2[2] = {al[0], al[1]};
                        mma8(d, h2, b2e[j], zero);
                        mma8(low[j], l2, b2e[j], low[j]);
                        mma8(low[j], m2, b2e[j], low[j]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[j][i] += d[i];
                }
            }
            // Pixels g and g + 8: padded columns g + 1 (odd for even g) and g + 9.
            uint8_t* o = p2 + ((y + 1) * T2_ROW + ((g & 1) ? (g + 1) >> 1 : T2_O + (g >> 1))) * 16 + 4 * t4;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    store3(o + 64 * i + j * T2_PLANE, 2 * T2_PLANE, relu(acc[j][2 * i] + low[j][2 * i] + bb2[2 * j]),
                           relu(acc[j][2 * i + 1] + low[j][2 * i + 1] + bb2[2 * j + 1]));
            }
        }
        __syncthreads();
        // Layer 3: two output rows of 8 pixels per warp; their sums for the mean.
        if (warp < 4) {
            float acc[2][4] = {}, lm[2][4] = {}, lw[2][4] = {};
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const uint32_t a0 = a3base + (uint32_t)(((k / 3) * T2_ROW + (k % 3 == 1 ? T2_O : (k % 3) >> 1)) * 16);
                uint32_t ah[4], am[4], al[4];
                ldsm4(ah, a0);
                ldsm4(am, a0 + 2 * T2_PLANE);
                ldsm4(al, a0 + 4 * T2_PLANE);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint2 w3 = b3[(2 * k + j) * 32 + lane];
                    const uint32_t b[2] = {w3.x, w3.y};
                    float d[4];
                    mma16(d, ah, b, zero);
                    mma16(lm[j], am, b, lm[j]);
                    mma16(lw[j], al, b, lw[j]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[j][i] += d[i];
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float c0 = bb3[2 * j], c1 = bb3[2 * j + 1];
                float v0 = relu(acc[j][0] + (lm[j][0] + lw[j][0]) + c0) + relu(acc[j][2] + (lm[j][2] + lw[j][2]) + c0);
                float v1 = relu(acc[j][1] + (lm[j][1] + lw[j][1]) + c1) + relu(acc[j][3] + (lm[j][3] + lw[j][3]) + c1);
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, o);
                    v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, o);
                }
                if (g == 0) {
                    float* r = red + (par * 4 + warp) * C3 + 8 * j + 2 * t4;
                    r[0] = v0;
                    r[1] = v1;
                }
            }
        }
        last = t;
        t = tn;
    }
    __syncthreads();
    if (warp == 0 && last >= 0) {
        // Parity of the last tile: tiles alternate from 0.
        const int k = (last - (int)blockIdx.x) / (int)gridDim.x;
        finish(last, k & 1);
    }
}

// ---------------------------------------------------------------------------
// One training step's loss and gradient in one kernel.
//
// A patch's part of the gradient needs nothing from other patches: its logit
// gives dLoss/dlogit.  So a block takes a patch through forward, loss and
// backward with everything in shared memory (the activations used to go out to
// and back from global memory, 53 KB per patch, between three kernels), and the
// weight gradients of its patches stay in registers until the end.
//
// Every product runs on the tensor cores like the forward's: activations and
// their gradients as three exact bf16 parts, weights as they are.  Products of
// two split numbers keep the six part products down to 2^-16 (the rest is below
// an fp32 rounding); leading parts' sums leave the tensor cores every 16 terms.
// The gradient entering layer 3 is one number per channel times the ReLU mask,
//   d3[o][p] = s_o mask[o][p],  s_o = dlogit w_f[o] / 64,
// so the mask (exact in bf16) is the operand: dW3 = s_o (mask a2), and d2 is
// (dlogit / 64) times the mask's transposed convolution with w_f[o] w3, a
// product of two bf16 numbers, hence exact in two.  Transposed stride-2
// convolutions split by the parity of the pixel: each of the four classes is a
// small matrix product of 1, 2, 2 or 4 taps over neighbouring pixels.
//
// 16 warps, one block per SM.  Phases of a patch, a barrier after each:
//   1 layer 1 (and the previous patch's dW1)   2 layer 2   3 layer 3, mask, the
//   next patch's pixels   4 loss, dW3, d2      5 dW2, d1.
// dW2 lives as one 16 x 72 accumulator per warp (its pixel rows), dW3 as one or
// two 16 x 8 tiles per warp, dW1 as one 9 x 8 tile per warp (its pixel rows).
// Bound by the latency of the phases (issue 46 %, shared memory 54 %, tensor
// pipe 30 %).  2048 patches: 2000 us as three fp32 kernels (1674 of them the
// backward's scalar loops), 127 us here.  Against 64 bits (medians of 48 batches of
// the committed network; before, as fp32 kernels): gradient 1.6e-7 of its norm off
// (2.2e-7), by layer, weights and bias: 1.6e-7, 1.2e-7 (2.7e-7, 1.7e-7); 1.7e-7,
// 1.4e-7 (2.2e-7, 1.9e-7); 1.6e-7, 1.4e-7 (2.2e-7, 1.9e-7); head 1.4e-7, 2.7e-8
// (1.6e-7, 1.0e-7; its bias summed in fp32 atomics was 1.2e-7 off).  Loss 1.9e-8
// (3.3e-8; 24 batches).
constexpr int TR_THREADS = 512, TR_WARPS = TR_THREADS / 32;
constexpr int M3_ROW = 9, M3_PLANE = 9 * M3_ROW * 16;      // layer-3 mask: 8 x 8 pixels, a zero row and column; one channel half
constexpr int D2_ROW = 17, D2_PLANE = 17 * D2_ROW * 16;    // d2: 16 x 16 pixels, a zero row and column; one part and half
constexpr int D1_PLANE = 32 * 32 * 16;                     // d1: 32 rows of 16 even, then 16 odd columns; one part
constexpr int FR = 128;                                    // bytes of one fragment register of a warp
constexpr int TR_IN = 0, TR_P1 = TR_IN + 2 * TI_BYTES, TR_P2 = TR_P1 + 3 * T1_PLANE, TR_M3 = TR_P2 + 6 * T2_PLANE,
              TR_D2 = TR_M3 + 2 * M3_PLANE, TR_D1 = TR_D2 + 6 * D2_PLANE, TR_F2 = TR_D1 + 3 * D1_PLANE,
              TR_F3 = TR_F2 + 18 * FR, TR_FQ = TR_F3 + 36 * FR, TR_FT = TR_FQ + 72 * FR, TR_RED = TR_FT + 18 * FR,
              TR_SMEM = TR_RED + 2 * 4 * C3 * 4 + 64;
static_assert(TR_SMEM <= 227 * 1024, "shared memory of one block");
static_assert(TR_M3 % 16 == 0 && TR_D2 % 16 == 0 && TR_D1 % 16 == 0 && TR_F2 % 16 == 0, "16-byte rows for ldmatrix");

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(a)
                 : "memory");
}

__global__ void __launch_bounds__(TR_THREADS, 1)
k_train(const uint8_t* __restrict__ tiles, const float* __restrict__ labels, int n, float pos_weight,
        const __nv_bfloat16* __restrict__ wq, float* __restrict__ grad, double* __restrict__ loss) {
    extern __shared__ __align__(128) uint8_t tsm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    uint8_t* const p1 = tsm + TR_P1;
    uint8_t* const p2 = tsm + TR_P2;
    uint8_t* const m3 = tsm + TR_M3;
    uint8_t* const d2 = tsm + TR_D2;
    uint8_t* const d1 = tsm + TR_D1;
    float* const red = reinterpret_cast<float*>(tsm + TR_RED);  // [sums, counts][row pair][channel]
    const uint32_t sb = smem_addr(tsm);
    for (int i = tid; i < TR_F2 / 16; i += TR_THREADS) reinterpret_cast<uint4*>(tsm)[i] = make_uint4(0u, 0u, 0u, 0u);

    // ---- weight fragments, one word per lane, in shared memory
    {
        auto put = [&](int base, int f, uint32_t v) { reinterpret_cast<uint32_t*>(tsm + base + f * FR)[lane] = v; };
        for (int f = warp; f < 18; f += TR_WARPS) {  // layer 2: (channel half j, step s, register), the ninth tap last
            const int j = f / 9, k = f % 9, r = W2 + (8 * j + g) * C1 * 9 + 2 * t4 * 9;
            put(TR_F2, f, k < 8 ? pack_w(wq, r + k, r + 9 + k) : pack_w(wq, r + 8, r + 9 + 8));
        }
        for (int f = warp; f < 36; f += TR_WARPS) {  // layer 3: (half j, tap, register)
            const int j = f / 18, k = f % 18 / 2, h = f & 1;
            const int r = W3 + (8 * j + g) * C2 * 9 + (8 * h + 2 * t4) * 9;
            put(TR_F3, f, pack_w(wq, r + k, r + 9 + k));
        }
        for (int f = warp; f < 36; f += TR_WARPS) {  // w_f w3 for d2: (half j of c, tap, register), two parts
            const int j = f / 18, k = f % 18 / 2, o = 8 * (f & 1) + 2 * t4, c = 8 * j + g;
            uint32_t hi = 0u, lo = 0u;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float q = __bfloat162float(wq[WF + o + e]) * __bfloat162float(wq[W3 + ((o + e) * C2 + c) * 9 + k]);
                const float h = __uint_as_float(__float_as_uint(q) & 0xFFFF0000u);
                hi |= (__float_as_uint(h) >> 16) << (16 * e);
                lo |= (__float_as_uint(q - h) >> 16) << (16 * e);
            }
            put(TR_FQ, 2 * f, hi);
            put(TR_FQ, 2 * f + 1, lo);
        }
        for (int f = warp; f < 18; f += TR_WARPS) {  // w2 for d1: (tap, register), depth o, channel c = g
            const int k = f >> 1, o = 8 * (f & 1) + 2 * t4;
            put(TR_FT, f, pack_w(wq, W2 + (o * C1 + g) * 9 + k, W2 + ((o + 1) * C1 + g) * 9 + k));
        }
    }
    auto frag = [&](int base, int f) { return reinterpret_cast<const uint32_t*>(tsm + base + f * FR)[lane]; };
    uint32_t b1[2];
    {
        auto w1 = [&](int k) { return k < 12 && (k & 3) ? W1 + g * 9 + (k >> 2) * 3 + (k & 3) - 1 : -1; };
        b1[0] = pack_w(wq, w1(2 * t4), w1(2 * t4 + 1));
        b1[1] = pack_w(wq, w1(2 * t4 + 8), w1(2 * t4 + 9));
    }
    auto wv = [&](int i) { return __bfloat162float(wq[i]); };
    const float wf = wv(WF + (lane & 15)), bf = wv(BF);
    const float wfg[2] = {wv(WF + g), wv(WF + g + 8)};
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
    auto col1 = [](int kx) { return kx == 1 ? T1_O : kx >> 1; };  // E[x], O[x], E[x + 1]
    auto col2 = [](int kx) { return kx == 1 ? T2_O : kx >> 1; };

    // ---- accumulators over the block's patches
    float g2[9][4] = {}, g3[2][4] = {}, g1[4] = {}, gb2[2] = {}, gb1[2] = {};
    float gwf = 0.f, gb3 = 0.f, gbf = 0.f;
    double lsum = 0.0;  // thread 0

    auto load = [&](int t) {
        Patch P;
        P.p = tiles + (size_t)t * S0 * S0;
        P.x0 = P.y0 = P.w = P.h = P.pitch = 0;
        return load_chunk(P, tid & 255);
    };
    // dW1 of the patch in buffer b: 16 pixels of one row and parity per step, depth = pixels,
    // rows = taps, columns = channels.
    auto grad1 = [&](int b) {
        const uint32_t* const in = reinterpret_cast<const uint32_t*>(tsm + TR_IN + b * TI_BYTES);
        const int ky = g / 3, kx = g % 3;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int iy = 2 * warp + (i >> 1), par = i & 1;
            uint32_t bh[2], bm[2], bl[2];
            const uint32_t ba = sb + TR_D1 + (uint32_t)((iy * 32 + par * 16 + (lane & 15)) * 16);
            ldsm2t(bh, ba);
            ldsm2t(bm, ba + D1_PLANE);
            ldsm2t(bl, ba + 2 * D1_PLANE);
            // Pixel k of the step is column 2 k + par: input column 4 k + 2 par + kx - 1.
            auto taps = [&](int ty, int tx, int k0) {  // values for k0 and k0 + 1, packed
                const uint32_t* r = in + (2 * iy + ty) * TI_ROW + TI_X + par + 2 * k0 - (tx == 0 ? 1 : 0);
                return __byte_perm(r[0], r[2], tx == 1 ? 0x5410 : 0x7632);
            };
            uint32_t a[4] = {taps(ky, kx, 2 * t4), 0u, taps(ky, kx, 2 * t4 + 8), 0u};
            if (g == 0) {
                a[1] = taps(2, 2, 2 * t4);
                a[3] = taps(2, 2, 2 * t4 + 8);
            }
            float d[4], low[4];
            mma16(d, a, bh, zero);
            mma16(low, a, bl, zero);
            mma16(low, a, bm, low);
#pragma unroll
            for (int e = 0; e < 4; ++e) g1[e] += d[e] + low[e];
        }
    };

    int t = blockIdx.x, buf = 0;
    bool any = false;  // a patch was finished: its dW1 is pending (in buffer buf ^ 1)
    __syncthreads();
    if (t < n && tid < 256) stage_bf16(reinterpret_cast<uint32_t*>(tsm + TR_IN), tid, load(t));
    __syncthreads();
    for (; t < n; buf ^= 1) {
        const int tn = t + gridDim.x;
        uint4 pix = make_uint4(0u, 0u, 0u, 0u);
        if (tn < n && tid >= 256) pix = load(tn);
        const float label = __ldg(labels + t);
        // ---- 1: dW1 of the previous patch; layer 1
        if (any) grad1(buf ^ 1);
        {
            const uint32_t* const in = reinterpret_cast<const uint32_t*>(tsm + TR_IN + buf * TI_BYTES);
            const float bb[2] = {wv(B1 + 2 * t4), wv(B1 + 2 * t4 + 1)};
#pragma unroll 2
            for (int i = warp; i < 64; i += TR_WARPS) {
                const int y = i >> 1, h = i & 1;
                const uint32_t* r = in + (2 * y + (t4 >> 1)) * TI_ROW + TI_X - 1 + 2 * g + 16 * h + (t4 & 1);
                const uint32_t* r2 = in + (2 * y + 2) * TI_ROW + TI_X - 1 + 2 * g + 16 * h + t4;
                uint32_t a[4] = {r[0], r[1], 0u, 0u};
                if (t4 < 2) {
                    a[2] = r2[0];
                    a[3] = r2[1];
                }
                float d[4];
                mma16(d, a, b1, zero);
                uint8_t* o = p1 + ((y + 1) * T1_ROW + g + 8 * h) * 16 + 4 * t4;
                store3(o + T1_O * 16, T1_PLANE, relu(d[0] + bb[0]), relu(d[1] + bb[1]));  // even columns
                store3(o + 16, T1_PLANE, relu(d[2] + bb[0]), relu(d[3] + bb[1]));
            }
        }
        __syncthreads();
        // ---- 2: layer 2, one output row per warp
        {
            const uint32_t row = sb + TR_P1 + (uint32_t)(2 * warp * T1_ROW * 16);
            const int x = (lane & 7) + 8 * ((lane >> 3) & 1);
            float acc[2][4] = {}, low[2][4] = {};
#pragma unroll
            for (int s = 0; s < 5; ++s) {
                const int tap = s < 4 ? 2 * s + (lane >> 4) : 8;
                const uint32_t a0 = row + (uint32_t)(((tap / 3) * T1_ROW + col1(tap % 3) + x) * 16);
                if (s < 4) {
                    uint32_t ah[4], am[4], al[4];
                    ldsm4(ah, a0);
                    ldsm4(am, a0 + T1_PLANE);
                    ldsm4(al, a0 + 2 * T1_PLANE);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t b[2] = {frag(TR_F2, 9 * j + 2 * s), frag(TR_F2, 9 * j + 2 * s + 1)};
                        float d[4];
                        mma16(d, ah, b, zero);
                        mma16(low[j], al, b, low[j]);
                        mma16(low[j], am, b, low[j]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[j][i] += d[i];
                    }
                } else {
                    uint32_t ah[2], am[2], al[2];
                    ldsm2(ah, a0);
                    ldsm2(am, a0 + T1_PLANE);
                    ldsm2(al, a0 + 2 * T1_PLANE);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t b = frag(TR_F2, 9 * j + 8);
                        float d[4];
                        mma8(d, ah, b, zero);
                        mma8(low[j], al, b, low[j]);
                        mma8(low[j], am, b, low[j]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[j][i] += d[i];
                    }
                }
            }
            uint8_t* o = p2 + ((warp + 1) * T2_ROW + ((g & 1) ? (g + 1) >> 1 : T2_O + (g >> 1))) * 16 + 4 * t4;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float bb[2] = {wv(B2 + 8 * j + 2 * t4), wv(B2 + 8 * j + 2 * t4 + 1)};
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    store3(o + 64 * i + j * T2_PLANE, 2 * T2_PLANE, relu(acc[j][2 * i] + low[j][2 * i] + bb[0]),
                           relu(acc[j][2 * i + 1] + low[j][2 * i + 1] + bb[1]));
            }
        }
        __syncthreads();
        // ---- 3: layer 3 (warps 0..7: two rows, one channel half), its mask, channel sums and counts
        if (warp < 8) {
            const int j = warp & 1, y = 2 * (warp >> 1);
            const uint32_t a3 =
                sb + TR_P2 + (uint32_t)((lane >> 4) * T2_PLANE + (2 * (y + ((lane >> 3) & 1)) * T2_ROW + (lane & 7)) * 16);
            float acc[4] = {}, lm[4] = {}, lw[4] = {};
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const uint32_t a0 = a3 + (uint32_t)(((k / 3) * T2_ROW + col2(k % 3)) * 16);
                uint32_t ah[4], am[4], al[4];
                ldsm4(ah, a0);
                ldsm4(am, a0 + 2 * T2_PLANE);
                ldsm4(al, a0 + 4 * T2_PLANE);
                const uint32_t b[2] = {frag(TR_F3, 18 * j + 2 * k), frag(TR_F3, 18 * j + 2 * k + 1)};
                float d[4];
                mma16(d, ah, b, zero);
                mma16(lm, am, b, lm);
                mma16(lw, al, b, lw);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] += d[i];
            }
            float v[4], s[4];  // channels 2t, 2t + 1 of pixels (y, g), (y + 1, g)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = relu(acc[i] + (lm[i] + lw[i]) + wv(B3 + 8 * j + 2 * t4 + (i & 1)));
#pragma unroll
            for (int i = 0; i < 2; ++i)
                *reinterpret_cast<uint32_t*>(m3 + j * M3_PLANE + ((y + i) * M3_ROW + g) * 16 + 4 * t4) =
                    (v[2 * i] > 0.f ? 0x3F80u : 0u) | (v[2 * i + 1] > 0.f ? 0x3F800000u : 0u);
            s[0] = v[0] + v[2];
            s[1] = v[1] + v[3];
            s[2] = (v[0] > 0.f ? 1.f : 0.f) + (v[2] > 0.f ? 1.f : 0.f);
            s[3] = (v[1] > 0.f ? 1.f : 0.f) + (v[3] > 0.f ? 1.f : 0.f);
#pragma unroll
            for (int o = 4; o < 32; o <<= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) s[i] += __shfl_xor_sync(0xFFFFFFFFu, s[i], o);
            if (g == 0) {
                float* r = red + (warp >> 1) * C3 + 8 * j + 2 * t4;
                r[0] = s[0];
                r[1] = s[1];
                r[4 * C3] = s[2];
                r[4 * C3 + 1] = s[3];
            }
        } else if (tn < n) {
            stage_bf16(reinterpret_cast<uint32_t*>(tsm + TR_IN + (buf ^ 1) * TI_BYTES), tid - 256, pix);
        }
        __syncthreads();
        // ---- 4: logit, loss, dlogit (every warp); dW3; d2
        float dl;
        {
            const float* r = red + (lane & 15);
            const float gap = ((r[0] + r[C3]) + (r[2 * C3] + r[3 * C3])) * (1.f / 64.f);
            const float cnt = (r[4 * C3] + r[5 * C3]) + (r[6 * C3] + r[7 * C3]);
            float z = gap * wf;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
            z += bf;
            const float wt = label > 0.5f ? pos_weight : 1.f;
            const float sp = z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z));
            const float sg = 1.f / (1.f + expf(-z));
            dl = wt * (sg - label) / (float)n;
            if (tid == 0) lsum += (double)(wt * (sp - label * z));
            gwf += dl * gap;
            gb3 += dl * wf * (1.f / 64.f) * cnt;
            gbf += dl;
        }
        // dW3: tile i of (tap, half of c); depth = 16 pixels, two rows at a time.
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = warp + TR_WARPS * q;
            if (i >= 18) break;
            const int k = i >> 1, h = i & 1;
            float acc[4] = {}, low[4] = {};
#pragma unroll
            for (int y = 0; y < S3; y += 2) {
                // The mask transposed: rows = channels o, depth = pixels (y, x), (y + 1, x).
                uint32_t a[4], bh[2], bm[2], bl[2];
                ldsm4t(a, sb + TR_M3 +
                              (uint32_t)(((lane >> 3) & 1) * M3_PLANE + ((y + (lane >> 4)) * M3_ROW + (lane & 7)) * 16));
                const uint32_t b0 = sb + TR_P2 + (uint32_t)(h * T2_PLANE + ((2 * (y + ((lane >> 3) & 1)) + k / 3) * T2_ROW +
                                                                            col2(k % 3) + (lane & 7)) * 16);
                ldsm2t(bh, b0);
                ldsm2t(bm, b0 + 2 * T2_PLANE);
                ldsm2t(bl, b0 + 4 * T2_PLANE);
                float d[4];
                mma16(d, a, bh, zero);
                mma16(low, a, bl, low);
                mma16(low, a, bm, low);
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[e] += d[e];
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) g3[q][e] += dl * (1.f / 64.f) * wfg[e >> 1] * (acc[e] + low[e]);
        }
        // d2: pixels (2u + py, 2v + px), two rows u, half j of the channels; two
        // classes (py, px) per warp: (0, 0) and (1, 1), or (0, 1) and (1, 0).
        {
            const int u = 2 * (warp >> 2), j = (warp >> 1) & 1, c2nd = warp & 1;
            const uint32_t am = sb + TR_M3 + (uint32_t)((lane >> 4) * M3_PLANE +
                                                        ((u + ((lane >> 3) & 1)) * M3_ROW + (lane & 7)) * 16);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int py = c, px = c2nd ? 1 - c : c;
                float acc[4] = {}, low[4] = {};
                // Rows: even pixels take ky = 1; odd ones ky = 0 from row u + 1 and ky = 2 from row u.
                for (int ky = py ? 0 : 1; ky < 3; ky += 2)
                    for (int kx = px ? 0 : 1; kx < 3; kx += 2) {
                        uint32_t a[4];
                        ldsm4(a, am + (uint32_t)(((ky == 0 ? 1 : 0) * M3_ROW + (kx == 0 ? 1 : 0)) * 16));
                        const int f = 2 * (18 * j + 2 * (3 * ky + kx));
                        const uint32_t bh[2] = {frag(TR_FQ, f), frag(TR_FQ, f + 2)},
                                       bl[2] = {frag(TR_FQ, f + 1), frag(TR_FQ, f + 3)};
                        float d[4];
                        mma16(d, a, bh, zero);
                        mma16(low, a, bl, low);
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[e] += d[e];
                    }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int iy = 2 * (u + i) + py, ix = 2 * g + px;
                    // ReLU of layer 2: the leading part is zero where the activation is.
                    const uint32_t a2 = *reinterpret_cast<const uint32_t*>(
                        p2 + j * T2_PLANE + ((iy + 1) * T2_ROW + (px ? g + 1 : T2_O + g)) * 16 + 4 * t4);
                    const float v0 = (a2 & 0xFFFFu) ? dl * (1.f / 64.f) * (acc[2 * i] + low[2 * i]) : 0.f;
                    const float v1 = (a2 >> 16) ? dl * (1.f / 64.f) * (acc[2 * i + 1] + low[2 * i + 1]) : 0.f;
                    gb2[0] += v0;
                    gb2[1] += v1;
                    store3(d2 + j * D2_PLANE + (iy * D2_ROW + ix) * 16 + 4 * t4, 2 * D2_PLANE, v0, v1);
                }
            }
        }
        __syncthreads();
        // ---- 5: dW2 (depth = the 16 pixels of row `warp`), then d1 (row pairs 2u, 2u + 1, u = warp)
        {
            uint32_t ah[4], am[4], al[4];
            const uint32_t a0 = sb + TR_D2 + (uint32_t)(((lane >> 3) & 1) * D2_PLANE +
                                                        (warp * D2_ROW + (lane & 7) + 8 * (lane >> 4)) * 16);
            ldsm4t(ah, a0);
            ldsm4t(am, a0 + 2 * D2_PLANE);
            ldsm4t(al, a0 + 4 * D2_PLANE);
            const uint32_t b0 = sb + TR_P1 + (uint32_t)((2 * warp * T1_ROW + (lane & 15)) * 16);
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                uint32_t bh[2], bm[2], bl[2];
                const uint32_t ba = b0 + (uint32_t)(((k / 3) * T1_ROW + col1(k % 3)) * 16);
                ldsm2t(bh, ba);
                ldsm2t(bm, ba + T1_PLANE);
                ldsm2t(bl, ba + 2 * T1_PLANE);
                float d[4], low[4];
                mma16(d, ah, bh, zero);
                mma16(low, al, bh, zero);
                mma16(low, ah, bl, low);
                mma16(low, am, bm, low);
                mma16(low, am, bh, low);
                mma16(low, ah, bm, low);
#pragma unroll
                for (int e = 0; e < 4; ++e) g2[k][e] += d[e] + low[e];
            }
        }
        {
            float acc[4][4] = {}, low[4][4] = {};  // class 2 py + px
            const uint32_t a0 = sb + TR_D2 + (uint32_t)((lane >> 4) * D2_PLANE + (warp * D2_ROW + (lane & 15)) * 16);
#pragma unroll
            for (int dd = 0; dd < 4; ++dd) {  // d2 pixel (u + dy, v + dx)
                const int dy = dd >> 1, dx = dd & 1;
                uint32_t ah[4], am[4], al[4];
                const uint32_t aa = a0 + (uint32_t)((dy * D2_ROW + dx) * 16);
                ldsm4(ah, aa);
                ldsm4(am, aa + 2 * D2_PLANE);
                ldsm4(al, aa + 4 * D2_PLANE);
#pragma unroll
                for (int cl = 0; cl < 4; ++cl) {
                    const int py = cl >> 1, px = cl & 1;
                    if ((dy && !py) || (dx && !px)) continue;
                    const int ky = !py ? 1 : dy ? 0 : 2, kx = !px ? 1 : dx ? 0 : 2;
                    const uint32_t b[2] = {frag(TR_FT, 2 * (3 * ky + kx)), frag(TR_FT, 2 * (3 * ky + kx) + 1)};
                    float d[4];
                    mma16(d, ah, b, zero);
                    mma16(low[cl], al, b, low[cl]);
                    mma16(low[cl], am, b, low[cl]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[cl][e] += d[e];
                }
            }
#pragma unroll
            for (int cl = 0; cl < 4; ++cl) {
                const int iy = 2 * warp + (cl >> 1), px = cl & 1;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int v = g + 8 * i;
                    const uint32_t a1 = *reinterpret_cast<const uint32_t*>(
                        p1 + ((iy + 1) * T1_ROW + (px ? v + 1 : T1_O + v)) * 16 + 4 * t4);
                    const float v0 = (a1 & 0xFFFFu) ? acc[cl][2 * i] + low[cl][2 * i] : 0.f;
                    const float v1 = (a1 >> 16) ? acc[cl][2 * i + 1] + low[cl][2 * i + 1] : 0.f;
                    gb1[0] += v0;
                    gb1[1] += v1;
                    store3(d1 + (iy * 32 + px * 16 + v) * 16 + 4 * t4, D1_PLANE, v0, v1);
                }
            }
        }
        any = true;
        t = tn;
        __syncthreads();
    }
    if (any) grad1(buf ^ 1);

    // ---- the block's sums into the gradient.  dW3's tiles have one owner each; the others are summed over the
    // warps in shared memory first (the planes are free: every warp is past its last read after the barrier).
    __syncthreads();
    if (!any) return;
    // Per warp: dW2 [16][8][9], dW1 [8][9], db2 [16], db1 [8].
    constexpr int N2 = C2 * C1 * 9, N1 = C1 * 9, NS = N2 + N1 + C2 + C1;
    static_assert(TR_WARPS * NS * 4 <= TR_F2 - TR_P1, "the sums fit the planes");
    float* const sum = reinterpret_cast<float*>(tsm + TR_P1);
    float* const own = sum + warp * NS;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int o = g + 8 * (e >> 1), c = 2 * t4 + (e & 1);
#pragma unroll
        for (int k = 0; k < 9; ++k) own[(o * C1 + c) * 9 + k] = g2[k][e];
        if (o <= 8) own[N2 + c * 9 + o] = g1[e];  // rows of dW1: taps 0 .. 8
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = warp + TR_WARPS * q;
            if (i < 18) atomicAdd(grad + W3 + (o * C2 + 8 * (i & 1) + c) * 9 + (i >> 1), g3[q][e]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            gb2[i] += __shfl_xor_sync(0xFFFFFFFFu, gb2[i], o);
            gb1[i] += __shfl_xor_sync(0xFFFFFFFFu, gb1[i], o);
        }
        if (g == 0) {
            const int j = (warp >> 1) & 1;  // the half of the channels whose d2 this warp made
            own[N2 + N1 + 8 * j + 2 * t4 + i] = gb2[i];
            own[N2 + N1 + 8 * (1 - j) + 2 * t4 + i] = 0.f;
            own[N2 + N1 + C2 + 2 * t4 + i] = gb1[i];
        }
    }
    if (warp == 0) {
        if (lane < C3) {
            atomicAdd(grad + WF + lane, gwf);
            atomicAdd(grad + B3 + lane, gb3);
        }
        if (lane == 0) {
            atomicAdd(loss, lsum / (double)n);
            atomicAdd(loss + 1, (double)gbf);
        }
    }
    __syncthreads();
    for (int i = tid; i < NS; i += TR_THREADS) {
        float v = 0.f;
        for (int w = 0; w < TR_WARPS; ++w) v += sum[w * NS + i];
        const int at = i < N2 ? W2 + i : i < N2 + N1 ? W1 + i - N2 : i < N2 + N1 + C2 ? B2 + i - N2 - N1 : B1 + i - N2 - N1 - C2;
        atomicAdd(grad + at, v);
    }
}

__global__ void k_adam(float* __restrict__ master, __nv_bfloat16* __restrict__ wq, const float* __restrict__ g,
                       const double* __restrict__ g_last, float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                       float wd, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    const float gi = i == BF ? (float)*g_last : g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float upd = (mi / c1) / (sqrtf(vi / c2) + eps) + wd * master[i];
    const float w = master[i] - lr * upd;
    master[i] = w;
    wq[i] = __float2bfloat16_rn(w);
}

__global__ void k_round(const float* __restrict__ master, __nv_bfloat16* __restrict__ wq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) wq[i] = __float2bfloat16_rn(master[i]);
}

__global__ void k_bf16_to_f32(const __nv_bfloat16* __restrict__ wq, float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NP) out[i] = __bfloat162float(wq[i]);
}

uint32_t crc32(const uint8_t* p, size_t n) {
    uint32_t c = 0xFFFFFFFFu;
    for (size_t i = 0; i < n; ++i) {
        c ^= p[i];
        for (int k = 0; k < 8; ++k) c = (c >> 1) ^ (0xEDB88320u & (0u - (c & 1u)));
    }
    return ~c;
}

int fail(int code, const std::string& m) {
    ofk::set_last_error(m);
    return code;
}

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

// Blocks of the inference kernel: FWD_BLOCKS on every SM, at most one per tile.
int fwd_grid(int n) {
    const int m = FWD_BLOCKS * sm_count();
    return n < m ? n : m;
}

// Proposal mask of one listed image per block (see of_detect_learned).
__global__ void k_propose(const ofk::Img* __restrict__ imgs, const int32_t* __restrict__ list,
                          const int32_t* __restrict__ prefix, const float* __restrict__ logits,
                          uint8_t* __restrict__ pos, uint8_t* __restrict__ mask, float threshold, float min_conf,
                          int dilate, int32_t* __restrict__ stats) {
    __shared__ float red[32];
    __shared__ int fallback, nprop;
    const int j = blockIdx.x;
    const ofk::Img& I = imgs[list[j]];
    const int base = prefix[j], n = prefix[j + 1] - base;
    const int ptx = 4 * I.tiles_x;
    float conf = 0.f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float p = 1.f / (1.f + expf(-logits[base + i]));
        conf += fabsf(2.f * p - 1.f);
        pos[base + i] = (p >= threshold) ? 1 : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) conf += __shfl_xor_sync(0xFFFFFFFFu, conf, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = conf;
    if (threadIdx.x == 0) nprop = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        float c = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) c += red[w];
        fallback = n > 0 && c / (float)n < min_conf;
    }
    __syncthreads();
    int cnt = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        uint8_t on = 1;
        if (!fallback) {
            const int px = i % ptx, py = i / ptx;
            on = pos[base + i];
            if (dilate && !on) {
                for (int dy = -1; dy <= 1 && !on; ++dy)
                    for (int dx = -1; dx <= 1 && !on; ++dx) {
                        const int qx = px + dx, qy = py + dy;
                        if (qx >= 0 && qx < ptx && qy >= 0 && qy < I.tiles_y) on = pos[base + qy * ptx + qx];
                    }
            }
        }
        mask[base + i] = on;
        cnt += on;
    }
    atomicAdd(&nprop, cnt);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(&stats[0], n);
        atomicAdd(&stats[1], nprop);
        if (fallback) atomicAdd(&stats[2], 1);
    }
}

// Patches of every proposal tile of one image, tile-major.
__global__ void k_extract(const ofk::Img* __restrict__ imgs, int img, int border, uint8_t* __restrict__ dst, int n) {
    const ofk::Img& I = imgs[img];
    const int ptx = 4 * I.tiles_x;
    for (int t = blockIdx.x; t < n; t += gridDim.x) {
        const int x0 = I.tile_x0 + 32 * (t % ptx) - 16, y0 = border + 32 * (t / ptx) - 16;
        for (int i = threadIdx.x; i < S0 * S0; i += blockDim.x) {
            const int x = x0 + (i & 63), y = y0 + (i >> 6);
            dst[(size_t)t * S0 * S0 + i] =
                (x >= 0 && x < I.w && y >= 0 && y < I.h) ? I.img[(size_t)y * I.pitch + x] : (uint8_t)0;
        }
    }
}

}  // namespace tn

namespace ofk {
int launch_propose(const Img* imgs, const int32_t* list, const int32_t* prefix, int n_list, const float* logits,
                   uint8_t* pos, uint8_t* mask, float threshold, float min_conf, int dilate, int32_t* stats,
                   void* stream) {
    if (n_list <= 0) return OF_OK;
    tn::k_propose<<<n_list, 256, 0, (cudaStream_t)stream>>>(imgs, list, prefix, logits, pos, mask, threshold,
                                                            min_conf, dilate, stats);
    return cudaGetLastError() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "proposal launch failed");
}

int launch_extract(const Img* imgs, int img, int border, uint8_t* dst, int n, void* stream) {
    if (n <= 0) return OF_OK;
    tn::k_extract<<<n < 1024 ? n : 1024, 256, 0, (cudaStream_t)stream>>>(imgs, img, border, dst, n);
    return cudaGetLastError() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "extract launch failed");
}

// Forward over the proposal tiles of a batch (in place from the pyramid); items: the batch's 128 x 32 detect tiles.
int tcnn_forward_tiles(of_tcnn* N, const Img* imgs, const uint2* items, int n_tiles, float* logits, void* stream) {
    if (n_tiles <= 0) return OF_OK;
    tn::PatchSrc src{nullptr, imgs, items};
    tn::k_forward_fast<<<tn::fwd_grid(n_tiles), tn::FWD_THREADS, tn::FWD_SMEM, (cudaStream_t)stream>>>(
        src, n_tiles, N->w, logits);
    return cudaGetLastError() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "tile-net forward launch failed");
}
}  // namespace ofk

extern "C" {

of_tcnn* of_tcnn_create(uint64_t seed) {
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(tn::k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, tn::TR_SMEM);
        cudaFuncSetAttribute(tn::k_forward_fast, cudaFuncAttributeMaxDynamicSharedMemorySize, tn::FWD_SMEM);
        attr = true;
    }
    of_tcnn* N = new of_tcnn();
    cudaGetDevice(&N->device);
    const size_t b = sizeof(float) * tn::NP;
    if (cudaMalloc(&N->master, b) != cudaSuccess || cudaMalloc(&N->w, sizeof(__nv_bfloat16) * tn::NP) != cudaSuccess ||
        cudaMalloc(&N->grad, sizeof(float) * tn::GRAD_WORDS) != cudaSuccess || cudaMalloc(&N->m, b) != cudaSuccess ||
        cudaMalloc(&N->v, b) != cudaSuccess) {
        tn::fail(OF_ERR_CUDA, "tile-net allocation failed");
        of_tcnn_destroy(N);
        return nullptr;
    }
    // He-uniform initialisation from a 64-bit LCG (host), biases 0.
    std::vector<float> p(tn::NP, 0.f);
    uint64_t s = seed * 6364136223846793005ull + 1442695040888963407ull;
    auto uni = [&]() {
        s = s * 6364136223846793005ull + 1442695040888963407ull;
        return (float)((s >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
    };
    auto fill = [&](int off, int count, int fan_in) {
        const float a = std::sqrt(6.f / (float)fan_in);
        for (int i = 0; i < count; ++i) p[off + i] = a * uni();
    };
    fill(tn::W1, tn::C1 * 9, 9);
    fill(tn::W2, tn::C2 * tn::C1 * 9, tn::C1 * 9);
    fill(tn::W3, tn::C3 * tn::C2 * 9, tn::C2 * 9);
    fill(tn::WF, tn::C3, tn::C3);
    if (of_tcnn_set_params(N, p.data()) != OF_OK) {
        of_tcnn_destroy(N);
        return nullptr;
    }
    return N;
}

void of_tcnn_destroy(of_tcnn* N) {
    if (!N) return;
    for (void* q : {(void*)N->master, (void*)N->w, (void*)N->grad, (void*)N->m, (void*)N->v})
        if (q) cudaFree(q);
    delete N;
}

int of_tcnn_num_params(void) { return tn::NP; }

int of_tcnn_set_params(of_tcnn* N, const float* host) {
    if (!N || !host) return tn::fail(OF_ERR_ARG, "null argument");
    const size_t b = sizeof(float) * tn::NP;
    if (cudaMemcpy(N->master, host, b, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(N->m, 0, b) != cudaSuccess || cudaMemset(N->v, 0, b) != cudaSuccess ||
        cudaMemset(N->grad, 0, sizeof(float) * tn::GRAD_WORDS) != cudaSuccess)
        return tn::fail(OF_ERR_CUDA, "tile-net upload failed");
    tn::k_round<<<(tn::NP + 255) / 256, 256>>>(N->master, N->w);
    N->step = 0;
    return cudaDeviceSynchronize() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "tile-net rounding failed");
}

int of_tcnn_get_params(of_tcnn* N, int which, float* host) {
    if (!N || !host || which < 0 || which > 2) return tn::fail(OF_ERR_ARG, "bad arguments");
    const size_t b = sizeof(float) * tn::NP;
    cudaError_t e;
    if (which == 0) {
        e = cudaMemcpy(host, N->master, b, cudaMemcpyDeviceToHost);
    } else if (which == 2) {
        std::vector<float> g(tn::GRAD_WORDS);
        e = cudaMemcpy(g.data(), N->grad, sizeof(float) * tn::GRAD_WORDS, cudaMemcpyDeviceToHost);
        double last = 0.0;
        std::memcpy(&last, g.data() + tn::LOSS_AT + 2, sizeof(last));
        g[tn::BF] = (float)last;
        if (e == cudaSuccess) std::memcpy(host, g.data(), b);
    } else {
        float* tmp = nullptr;
        e = cudaMalloc(&tmp, b);
        if (e == cudaSuccess) {
            tn::k_bf16_to_f32<<<(tn::NP + 255) / 256, 256>>>(N->w, tmp);
            e = cudaMemcpy(host, tmp, b, cudaMemcpyDeviceToHost);
            cudaFree(tmp);
        }
    }
    return e == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "tile-net download failed");
}

int of_tcnn_forward(of_tcnn* N, const uint8_t* tiles, int n, float* logits, void* stream) {
    if (!N || !tiles || !logits || n < 0) return tn::fail(OF_ERR_ARG, "bad arguments");
    if (n == 0) return OF_OK;
    tn::PatchSrc src{tiles, nullptr, nullptr};
    tn::k_forward_fast<<<tn::fwd_grid(n), tn::FWD_THREADS, tn::FWD_SMEM, (cudaStream_t)stream>>>(src, n, N->w, logits);
    return cudaGetLastError() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "tile-net forward launch failed");
}

int of_tcnn_loss_grad(of_tcnn* N, const uint8_t* tiles, const float* labels, int n, float pos_weight,
                      float* loss_out, void* stream) {
    if (!N || !tiles || !labels || n < 1 || !(pos_weight > 0.f)) return tn::fail(OF_ERR_ARG, "bad arguments");
    cudaStream_t st = (cudaStream_t)stream;
    double* const loss = reinterpret_cast<double*>(N->grad + tn::LOSS_AT);
    cudaMemsetAsync(N->grad, 0, sizeof(float) * tn::GRAD_WORDS, st);
    const int sms = tn::sm_count();
    tn::k_train<<<n < sms ? n : sms, tn::TR_THREADS, tn::TR_SMEM, st>>>(tiles, labels, n, pos_weight, N->w, N->grad, loss);
    if (cudaGetLastError() != cudaSuccess) return tn::fail(OF_ERR_CUDA, "tile-net training launch failed");
    if (loss_out) {
        double sum = 0.0;
        if (cudaMemcpyAsync(&sum, loss, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return tn::fail(OF_ERR_CUDA, "tile-net loss readback failed");
        *loss_out = (float)sum;
    }
    return OF_OK;
}

int of_tcnn_adam(of_tcnn* N, float lr, float beta1, float beta2, float eps, float weight_decay, void* stream) {
    if (!N || !(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f))
        return tn::fail(OF_ERR_ARG, "bad Adam arguments");
    N->step += 1;
    const float c1 = 1.f - std::pow(beta1, (float)N->step), c2 = 1.f - std::pow(beta2, (float)N->step);
    const double* const last = reinterpret_cast<const double*>(N->grad + tn::LOSS_AT) + 1;
    tn::k_adam<<<(tn::NP + 255) / 256, 256, 0, (cudaStream_t)stream>>>(N->master, N->w, N->grad, last, N->m, N->v, lr,
                                                                        beta1, beta2, eps, weight_decay, c1, c2);
    return cudaGetLastError() == cudaSuccess ? OF_OK : tn::fail(OF_ERR_CUDA, "Adam launch failed");
}

// Checkpoint: "OFTC" | version u32 | n_params u32 | step i64 | master | m | v | crc32 of all before it.
int64_t of_tcnn_save(of_tcnn* N, uint8_t* buf, int64_t cap) {
    if (!N) return tn::fail(OF_ERR_ARG, "null net");
    const size_t body = 4 + 4 + 4 + 8 + 3 * sizeof(float) * tn::NP;
    const int64_t total = (int64_t)body + 4;
    if (!buf) return total;
    if (cap < total) return tn::fail(OF_ERR_ARG, "buffer too small");
    std::vector<float> a(tn::NP), m(tn::NP), v(tn::NP);
    if (cudaMemcpy(a.data(), N->master, sizeof(float) * tn::NP, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(m.data(), N->m, sizeof(float) * tn::NP, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(v.data(), N->v, sizeof(float) * tn::NP, cudaMemcpyDeviceToHost) != cudaSuccess)
        return tn::fail(OF_ERR_CUDA, "download failed");
    uint8_t* p = buf;
    std::memcpy(p, "OFTC", 4);
    const uint32_t ver = 1, np = tn::NP;
    std::memcpy(p + 4, &ver, 4);
    std::memcpy(p + 8, &np, 4);
    std::memcpy(p + 12, &N->step, 8);
    std::memcpy(p + 20, a.data(), sizeof(float) * tn::NP);
    std::memcpy(p + 20 + sizeof(float) * tn::NP, m.data(), sizeof(float) * tn::NP);
    std::memcpy(p + 20 + 2 * sizeof(float) * tn::NP, v.data(), sizeof(float) * tn::NP);
    const uint32_t crc = tn::crc32(buf, body);
    std::memcpy(p + body, &crc, 4);
    return total;
}

int of_tcnn_load(of_tcnn* N, const uint8_t* buf, int64_t n) {
    if (!N || !buf) return tn::fail(OF_ERR_ARG, "null argument");
    const size_t body = 4 + 4 + 4 + 8 + 3 * sizeof(float) * tn::NP;
    if (n != (int64_t)body + 4) return tn::fail(OF_ERR_ARG, "checkpoint size mismatch");
    uint32_t ver, np, crc;
    std::memcpy(&ver, buf + 4, 4);
    std::memcpy(&np, buf + 8, 4);
    std::memcpy(&crc, buf + body, 4);
    if (std::memcmp(buf, "OFTC", 4) != 0 || ver != 1 || np != (uint32_t)tn::NP)
        return tn::fail(OF_ERR_ARG, "not a version-1 tile-net checkpoint");
    if (tn::crc32(buf, body) != crc) return tn::fail(OF_ERR_ARG, "checkpoint CRC mismatch");
    const int rc = of_tcnn_set_params(N, reinterpret_cast<const float*>(buf + 20));
    if (rc != OF_OK) return rc;
    std::memcpy(&N->step, buf + 12, 8);
    if (cudaMemcpy(N->m, buf + 20 + sizeof(float) * tn::NP, sizeof(float) * tn::NP, cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(N->v, buf + 20 + 2 * sizeof(float) * tn::NP, sizeof(float) * tn::NP, cudaMemcpyHostToDevice) !=
            cudaSuccess)
        return tn::fail(OF_ERR_CUDA, "upload failed");
    return OF_OK;
}

}  // extern "C"
