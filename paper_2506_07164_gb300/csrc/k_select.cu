// Top-N per level: keep the n_l best NMS survivors of each (frame, level)
// image -- Harris key descending, then y ascending, then x ascending (Harris
// "screens" the FAST points, Sec. 1 and Sec. 3.2) -- as a list that is either
// in rank order or grouped by key code, better codes first (select_grouped).
//
// Each candidate has a unique 96-bit rank word
//   R = (key ^ 2^63) << 32 | ~((y << 16) | x),
// larger R = better rank.  A 4096-bin histogram of a code of the key that is
// monotone in the key (sign, bit length and the next 5 bits of |key|) locates the
// bin b holding the n_l-th largest key.  Then
//   - sorted list: every candidate with code >= b is gathered and sorted, and the
//     first n_l are kept;
//   - grouped list: candidates with code > b go straight to the places that the
//     counts of the better bins give them; those of bin b go through the same step
//     once more, by the next 9 bits of |key|, and the few of that boundary are
//     ranked by counting.
// A bin b that holds too many for that (the sort buffer, or SEL_BND) is narrowed
// first, by 12 bits of R at a time from the highest bit in which its candidates
// differ: one round for most 4K frames that need it; equal keys, say of a printed
// grid, go straight to the bits of their positions.  (By an MSB-first radix select
// of one block instead: some 4K frames 324 us a call, 205 so; a 1080p grid, 8192
// features, 256 us for the stage, 39 so.)
// Sorted lists are bitonic-sorted by R, descending; strides below 64 run in a
// warp's registers (shuffles), the rest through shared memory.
//
// The scans are latency-bound: a 1080p level 0 holds ~43 k candidates, a 4K
// one ~170 k, and one block scanning them twice set the whole stage's length
// (41 us for one 1080p frame, 131 us at 4K; now 16 and 27 us, of which ~8 us
// are the measurement's own launch and events).  So a cluster of C blocks
// shares an image: every block histograms and gathers its part of the
// candidates, block r sums bins [4096 r / C, ...) of all C histograms through
// distributed shared memory, and the gathered entries go to the first block.
// Every scan keeps SEL_UNROLL 16-byte loads (two keys) in flight per thread;
// the positions of the gathered candidates only are read.  Images with few
// candidates are left to the first block.  The sort is one block's chain of
// barriers (of 1000 keypoints: 5 of 21 us with one 1080p frame, of 8192: 35 of
// 49), while the orientation kernel has a warp for each keypoint: it finds the
// ranks of grouped lists.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "of_internal.h"
#include "of_launch.cuh"
#include "of_rank.cuh"

namespace ofk {

constexpr int SEL_UNROLL = 4;   // candidates loaded per thread before use
constexpr int SEL_BINS = 4096;  // coarse-pass histogram bins
constexpr int SEL_SOLO = 4096;  // candidates one block scans alone (one round of its loads)
constexpr int SEL_SOLO_G = 8192;  // ... of a grouped list (no sort beside it)
constexpr int SEL_MIN_SORT = 64;  // entries of the smallest sort (one warp's registers)
constexpr int SEL_MAX_DYN = 192 * 1024;
constexpr int SEL_BND = 2048;   // grouped lists: candidates of the boundary bin the first block takes
constexpr int SEL_RANK = 128;   // ... and ranks by counting

struct SelState {
    int coarse, code_b;  // the boundary bin fits; its code
    int n_take;          // grouped: candidates above the bin; sorted: those and the bin's
    int at;              // sorted: where a block's entries go in the first block's list
    int split, sure;     // the bin was narrowed to the prefix; its candidates above that
    uint64_t pre_hi, msk_hi;
    uint32_t pre_lo, msk_lo;
};

// The 9 bits of the magnitude after those of the code, for keys of one code:
// non-decreasing in key.
__device__ __forceinline__ uint32_t fine_bits(uint64_t u) {
    const bool pos = (u >> 63) != 0;
    const uint64_t x = pos ? u & 0x7FFFFFFFFFFFFFFFull : u ^ 0x7FFFFFFFFFFFFFFFull;
    const uint32_t f = x ? (uint32_t)((x << __clzll((long long)x) << 6) >> 55) : 0u;
    return pos ? f : 511u - f;
}

// The N bits of rank words that start at the highest bit in which some of them
// differ: `all` and `any` are their AND and OR as three words, highest first.
template <int N>
struct RankDigit {
    int sh;  // the digit is bits sh .. sh + N - 1 of the 96; the words agree above
    __device__ __forceinline__ RankDigit(const uint32_t* all, const uint32_t* any) {
        const uint32_t d0 = all[0] ^ any[0], d1 = all[1] ^ any[1], d2 = all[2] ^ any[2];
        const int p = d0 ? 95 - __clz(d0) : d1 ? 63 - __clz(d1) : 31 - __clz(d2);
        sh = max(p - N + 1, 0);
    }
    __device__ __forceinline__ uint32_t of(uint64_t hi, uint32_t lo) const {
        return (uint32_t)(sh >= 32 ? hi >> (sh - 32) : hi << (32 - sh) | lo >> sh) & ((1u << N) - 1u);
    }
};
// AND (words 0 .. 2) and OR (3 .. 5) of the warps' rank words into `bits`, preset to ones and zeros.
__device__ __forceinline__ void merge_bits(uint32_t* bits, const uint32_t (&all)[3], const uint32_t (&any)[3], int lane) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const uint32_t a = __reduce_and_sync(0xFFFFFFFFu, all[j]), o = __reduce_or_sync(0xFFFFFFFFu, any[j]);
        if (lane == 0) {
            atomicAnd(&bits[j], a);
            atomicOr(&bits[3 + j], o);
        }
    }
}

// ---- cluster primitives (shared::cluster addresses of the other blocks' shared memory)
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
// The address of this block's shared variable p in block `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_rank(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void st_rank(uint32_t a, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void st_rank64(uint32_t a, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ int atomic_add_rank(uint32_t a, int v) {
    int o;
    asm volatile("atom.relaxed.cluster.shared::cluster.add.s32 %0, [%1], %2;" : "=r"(o) : "r"(a), "r"(v) : "memory");
    return o;
}

// Bitonic sort of P entries (a power of two, at least 64), descending by
// (key, ~yx).  A warp keeps 64 consecutive entries in registers, two per lane
// (lane, lane + 32), for every stride below 64; longer strides go through
// shared memory, one thread per compared pair.
__device__ __forceinline__ void sort_cx(uint64_t& k, uint32_t& y, int j, bool want_max) {
    const uint64_t ok = __shfl_xor_sync(0xFFFFFFFFu, k, j);
    const uint32_t oy = __shfl_xor_sync(0xFFFFFFFFu, y, j);
    if (rank_less(k, ~y, ok, ~oy) == want_max) {
        k = ok;
        y = oy;
    }
}

// Strides min(k / 2, 32) .. 1 of stage k for the 64 entries from `base`.
__device__ __forceinline__ void sort_seg_stage(uint64_t (&e)[2], uint32_t (&y)[2], int base, int lane, int k) {
    if (k >= 64) {
        const bool desc = ((base + lane) & k) == 0;
        if (rank_less(e[0], ~y[0], e[1], ~y[1]) == desc) {
            const uint64_t te = e[0];
            const uint32_t ty = y[0];
            e[0] = e[1];
            y[0] = y[1];
            e[1] = te;
            y[1] = ty;
        }
    }
    for (int j = k >= 64 ? 16 : k >> 1; j > 0; j >>= 1) {
        const bool lower = (lane & j) == 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool desc = ((base + 32 * h + lane) & k) == 0;
            sort_cx(e[h], y[h], j, lower == desc);
        }
    }
}

__device__ __forceinline__ void bitonic_sort(uint64_t* skey, uint32_t* syx, int P, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    auto segments = [&](auto&& stages) {
        for (int base = 64 * warp; base < P; base += 2 * SELECT_THREADS) {
            uint64_t e[2] = {skey[base + lane], skey[base + 32 + lane]};
            uint32_t y[2] = {syx[base + lane], syx[base + 32 + lane]};
            stages(e, y, base);
            skey[base + lane] = e[0];
            skey[base + 32 + lane] = e[1];
            syx[base + lane] = y[0];
            syx[base + 32 + lane] = y[1];
        }
        __syncthreads();
    };
    segments([&](uint64_t(&e)[2], uint32_t(&y)[2], int base) {
        for (int k = 2; k <= 64; k <<= 1) sort_seg_stage(e, y, base, lane, k);
    });
    for (int k = 128; k <= P; k <<= 1) {
        for (int jj = k >> 1; jj >= 64; jj >>= 1) {
            for (int p = tid; p < (P >> 1); p += SELECT_THREADS) {
                const int i = ((p & ~(jj - 1)) << 1) | (p & (jj - 1));
                const int l = i | jj;
                const uint64_t ah = skey[i], bh = skey[l];
                const uint32_t ay = syx[i], by = syx[l];
                if (rank_less(ah, ~ay, bh, ~by) == ((i & k) == 0)) {
                    skey[i] = bh;
                    skey[l] = ah;
                    syx[i] = by;
                    syx[l] = ay;
                }
            }
            __syncthreads();
        }
        segments([&](uint64_t(&e)[2], uint32_t(&y)[2], int base) { sort_seg_stage(e, y, base, lane, k); });
    }
}

// Sum over the block's threads after this one.
__device__ __forceinline__ int threads_after(int own, uint32_t* wsum, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    int v = own;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int t = __shfl_down_sync(0xFFFFFFFFu, v, off);
        if (lane + off < 32) v += t;
    }
    if (lane == 0) wsum[warp] = (uint32_t)v;
    __syncthreads();
    int above = v - own;
    for (int w = warp + 1; w < SELECT_THREADS / 32; ++w) above += (int)wsum[w];
    return above;
}

// What the narrowing of ties shares: AND and OR of rank words (the block's, the
// cluster's), a split's boundary digit, the number needed of it and held by it.
struct TieState {
    uint32_t bits[6], all[6];
    int pick[3];
};

// A boundary bin that holds too many: the cluster narrows it, 12 bits of the rank
// words at a time from the highest bit in which its candidates differ (equal keys
// differ in their positions), until those that share the boundary's prefix fit --
// at most SEL_BND for the first block to rank (GROUPED), or as many as the sort
// buffer (cap) holds beside the better ones.  n_above: candidates above the bin;
// h2: SEL_BINS counts.
template <int C, bool GROUPED>
__device__ __forceinline__ void narrow_bin(const uint64_t* ckey, const uint32_t* cyx, int n, int parts, int q, int n_above,
                                        int cap, uint32_t* h2, uint32_t* wsum, TieState& T, SelState& st, int* s_cnt) {
    const int tid = threadIdx.x, lane = tid & 31, rank = (int)(blockIdx.x % C);
    const bool shared = parts > 1;
    const int i_first = rank * SELECT_THREADS + tid, i_step = parts * SELECT_THREADS;
    const uint32_t code_b = (uint32_t)st.code_b;
    const int need0 = q - n_above;
    int need = need0, left = 0;
    uint64_t pre_hi = 0ull, msk_hi = 0ull;
    uint32_t pre_lo = 0u, msk_lo = 0u;
    auto sync = [&] {
        if (shared) cluster_sync_all();
        else __syncthreads();
    };
    auto each = [&](auto&& f) {  // this block's candidates of the bin with the prefix
        for (int i0 = i_first; i0 < n; i0 += SEL_UNROLL * i_step) {
            uint64_t hi[SEL_UNROLL];
            uint32_t lo[SEL_UNROLL];
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
                hi[k] = i < n ? ckey[i] : 0ull;
                lo[k] = i < n ? ~cyx[i] : 0u;
            }
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k)
                if (i0 + k * i_step < n && key_code(hi[k]) == code_b && (hi[k] & msk_hi) == pre_hi &&
                    (lo[k] & msk_lo) == pre_lo)
                    f(hi[k], lo[k]);
        }
    };
    for (int round = 0; round < 8; ++round) {  // 12 of 96 bits a round
        if (tid < 6) T.bits[tid] = tid < 3 ? 0xFFFFFFFFu : 0u;
        if (tid < 3) T.pick[tid] = 0;  // ends the loop in all blocks alike
        for (int i = tid; i < SEL_BINS; i += SELECT_THREADS) h2[i] = 0u;
        __syncthreads();
        uint32_t all[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, any[3] = {0u, 0u, 0u};
        each([&](uint64_t hi, uint32_t lo) {
            const uint32_t w[3] = {(uint32_t)(hi >> 32), (uint32_t)hi, lo};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                all[j] &= w[j];
                any[j] |= w[j];
            }
        });
        merge_bits(T.bits, all, any, lane);
        sync();
        if (tid < 6) {
            uint32_t v = T.bits[tid];
            for (int c = 0; c < parts && shared; ++c) {
                const uint32_t o = ld_rank(map_rank(&T.bits[tid], c));
                v = tid < 3 ? v & o : v | o;
            }
            T.all[tid] = v;
        }
        __syncthreads();
        const RankDigit<12> dg(T.all, T.all + 3);
        each([&](uint64_t hi, uint32_t lo) { atomicAdd(&h2[dg.of(hi, lo)], 1u); });
        sync();
        if (rank == 0) {
            constexpr int PER1 = SEL_BINS / SELECT_THREADS;
            int bins[PER1], own = 0;
#pragma unroll
            for (int j = 0; j < PER1; ++j) {
                uint32_t h = 0u;
                for (int c = 0; c < parts; ++c) h += shared ? ld_rank(map_rank(&h2[PER1 * tid + j], c)) : h2[PER1 * tid + j];
                bins[j] = (int)h;
                own += (int)h;
            }
            const int above = threads_after(own, wsum, tid);
            if (above < need && above + own >= need) {  // exactly one thread
                int cum = above;
#pragma unroll
                for (int j = PER1 - 1; j >= 0; --j) {
                    if (cum < need && cum + bins[j] >= need) {
                        const int pick[3] = {PER1 * tid + j, need - cum, bins[j]};
                        for (int c = 0; c < parts; ++c)
                            for (int e = 0; e < 3; ++e) {
                                if (c == 0) T.pick[e] = pick[e];
                                else st_rank(map_rank(&T.pick[e], c), (uint32_t)pick[e]);
                            }
                    }
                    cum += bins[j];
                }
            }
        }
        sync();
        // The words agree above the digit: the prefix is their common bits and the digit.
        const uint64_t d = (uint64_t)T.pick[0];
        need = T.pick[1];
        left = T.pick[2];
        const int sh = dg.sh;
        const uint64_t common = (uint64_t)T.all[0] << 32 | T.all[1];
        if (sh >= 32) {
            msk_hi = ~0ull << (sh - 32);
            pre_hi = (common & ~(0xFFFull << (sh - 32)) & msk_hi) | d << (sh - 32);
        } else {
            msk_hi = ~0ull;
            pre_hi = (common & ~(0xFFFull >> (32 - sh))) | d >> (32 - sh);
            msk_lo = ~0u << sh;
            pre_lo = (T.all[2] & ~(0xFFFu << sh) & msk_lo) | (uint32_t)d << sh;
        }
        __syncthreads();
        if (left <= (GROUPED ? SEL_BND : cap - (q - need))) break;  // the same in all blocks
    }
    if (tid == 0) {
        st.pre_hi = pre_hi;
        st.msk_hi = msk_hi;
        st.pre_lo = pre_lo;
        st.msk_lo = msk_lo;
        st.sure = need0 - need;
        st.split = 1;
        st.coarse = 1;
        if (GROUPED) *s_cnt = n_above;  // where the bin's sure ones go
        else st.n_take = q - need + left;
    }
    sync();
}

// Apart from the code of grouped lists, whose images mostly run through without it
// (inside it a single frame's call took 0.5 us longer; sorted lists keep their
// registers better with it inside).
template <int C>
__device__ __noinline__ void narrow_bin_apart(const uint64_t* ckey, const uint32_t* cyx, int n, int parts, int q, int n_above,
                                              int cap, uint32_t* h2, uint32_t* wsum, TieState& T, SelState& st, int* s_cnt) {
    narrow_bin<C, true>(ckey, cyx, n, parts, q, n_above, cap, h2, wsum, T, st, s_cnt);
}

// The first block's boundary candidates `left` (nl of them, the best one's place
// `base`): while they are more than SEL_RANK they are narrowed by 9 bits of their
// rank words at a time, the better ones kept; the rest is ranked by counting.
__device__ __noinline__ void rank_ties(const uint64_t* bkey, const uint32_t* byx, uint32_t* hist, uint16_t* left, int nl,
                                       int base, int q, uint32_t* wsum, TieState& T, int* s_left, int* s_cnt, int* s_fine,
                                       uint64_t* kkey, uint32_t* kyx) {
    const int tid = threadIdx.x, lane = tid & 31;
    uint16_t* next = reinterpret_cast<uint16_t*>(hist + 2048);
    static_assert(2 * SEL_BND <= 4 * 1024, "room for the lists behind the 512 counts");
    for (int round = 0; nl > SEL_RANK && round < 11; ++round) {
        if (tid < 6) T.bits[tid] = tid < 3 ? 0xFFFFFFFFu : 0u;
        hist[tid] = 0u;
        if (tid == 0) {
            *s_left = 0;
            *s_cnt = base;
        }
        __syncthreads();
        uint32_t all[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, any[3] = {0u, 0u, 0u};
        for (int i = tid; i < nl; i += SELECT_THREADS) {
            const uint64_t hi = bkey[left[i]];
            const uint32_t w[3] = {(uint32_t)(hi >> 32), (uint32_t)hi, ~byx[left[i]]};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                all[j] &= w[j];
                any[j] |= w[j];
            }
        }
        merge_bits(T.bits, all, any, lane);
        __syncthreads();
        const RankDigit<9> dg(T.bits, T.bits + 3);
        for (int i = tid; i < nl; i += SELECT_THREADS) atomicAdd(&hist[dg.of(bkey[left[i]], ~byx[left[i]])], 1u);
        __syncthreads();
        const int own = (int)hist[tid], better = threads_after(own, wsum, tid);
        if (base + better < q && base + better + own >= q) *s_fine = tid | better << 9;
        __syncthreads();
        const int fine = *s_fine & 511;
        for (int i = tid; i < nl; i += SELECT_THREADS) {
            const int e = left[i], c = (int)dg.of(bkey[e], ~byx[e]);
            if (c > fine) {
                const int pos = atomicAdd(s_cnt, 1);
                if (pos < q) {
                    kkey[pos] = bkey[e];
                    kyx[pos] = byx[e];
                }
            } else if (c == fine) {
                next[atomicAdd(s_left, 1)] = (uint16_t)e;
            }
        }
        __syncthreads();
        base += *s_fine >> 9;
        nl = *s_left;
        uint16_t* const t = left;
        left = next;
        next = t;
        __syncthreads();
    }
    for (int i = tid; i < nl; i += SELECT_THREADS) {
        const uint64_t key = bkey[left[i]];
        const uint32_t yx = byx[left[i]];
        int place = base;
        for (int j = 0; j < nl; ++j) place += rank_less(key, ~yx, bkey[left[j]], ~byx[left[j]]);
        if (place < q) {
            kkey[place] = key;
            kyx[place] = yx;
        }
    }
}

// (Three blocks per SM of sorted lists, whose launches hold many images; grouped ones have no such bound.)
template <int C, bool GROUPED>
__global__ void __launch_bounds__(SELECT_THREADS, GROUPED ? 0 : 3)
k_select(const Img* __restrict__ imgs, const Call* __restrict__ call, int sort_cap) {
    extern __shared__ __align__(16) uint8_t dyn[];
    __shared__ uint32_t hist[SEL_BINS];
    __shared__ uint32_t wsum[SELECT_THREADS / 32];
    __shared__ uint32_t slice_sum[C];  // candidates in each block's slice of the bins
    __shared__ SelState st;
    __shared__ int s_cnt;
    __shared__ uint64_t bkey[GROUPED ? SEL_BND : 1];  // the boundary bin's candidates (first block)
    __shared__ uint32_t byx[GROUPED ? SEL_BND : 1];
    __shared__ int s_bnd, s_left, s_fine;  // their number, that of the fine boundary bin, its code
    __shared__ TieState tie;

    const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;  // block's place in its image's cluster
    // Images are stored frame by frame; a grid of two dimensions takes them level by level.
    const Img& I = imgs[blockIdx.x / C * gridDim.y + blockIdx.y];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = I.quota;
    const int32_t* const ctr = I.ctr;
    pdl_trigger();
    for (int i = tid; i < SEL_BINS; i += SELECT_THREADS) hist[i] = 0u;
    pdl_wait();  // the candidates
    const int n = min(ctr[0], I.cand_cap);
    if (q <= 0 || n <= 0) {  // the same for all blocks of the cluster
        if (tid == 0 && rank == 0) I.ctr[1] = 0;
        return;
    }
    // Blocks that share the scan: all of the cluster, or only the first.
    const bool shared = C > 1 && (GROUPED || n > q) && n > (GROUPED ? SEL_SOLO_G : SEL_SOLO);
    if (rank != 0 && !shared) return;
    const int parts = shared ? C : 1;
    const int m = min(n, q);
    uint64_t* skey = reinterpret_cast<uint64_t*>(dyn);
    uint32_t* syx = reinterpret_cast<uint32_t*>(dyn + sizeof(uint64_t) * (size_t)sort_cap);

    if (tid == 0) {
        st.coarse = n <= q;  // everything is kept: no boundary bin
        st.code_b = GROUPED ? -1 : 0;
        st.n_take = m;
        st.split = 0;
        st.sure = 0;
        s_cnt = 0;
        s_bnd = 0;
    }
    __syncthreads();

    // This block's candidate pairs: first, step (in pairs of keys).
    const int i_first = rank * SELECT_THREADS + tid, i_step = parts * SELECT_THREADS;
    if (GROUPED || n > q) {
        // Coarse pass: histogram of the key code, two keys per 16-byte load
        // (the candidate arrays start on 256-byte boundaries).
        const ulonglong2* ck2 = reinterpret_cast<const ulonglong2*>(I.ckey);
        const int n2 = n >> 1;
        for (int i0 = i_first; i0 < n2; i0 += SEL_UNROLL * i_step) {
            ulonglong2 v[SEL_UNROLL];
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
                v[k] = i < n2 ? ck2[i] : make_ulonglong2(0ull, 0ull);
            }
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k)
                if (i0 + k * i_step < n2) {
                    atomicAdd(&hist[key_code(v[k].x)], 1u);
                    atomicAdd(&hist[key_code(v[k].y)], 1u);
                }
        }
        if ((n & 1) && tid == 0 && rank == 0) atomicAdd(&hist[key_code(I.ckey[n - 1])], 1u);
        if (shared) cluster_sync_all();
        else __syncthreads();
        // Suffix sums: higher bins = better keys.  Shared scan: block r owns
        // bins [4096 r / C, +4096 / C) of the summed histograms, thread t
        // PER = 8 / C of them; else the block's thread t owns bins [8t, 8t + 8).
        constexpr int PER1 = SEL_BINS / SELECT_THREADS, PER = PER1 / C;
        int bins[PER1];
        int own = 0, b0, per;
        if (shared) {
            per = PER;
            b0 = rank * (SEL_BINS / C) + tid * PER;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                uint32_t h = 0u;
#pragma unroll
                for (int c = 0; c < C; ++c) h += ld_rank(map_rank(&hist[b0 + j], c));
                bins[j] = (int)h;
                own += (int)h;
            }
        } else {
            per = PER1;
            b0 = tid * PER1;
#pragma unroll
            for (int j = 0; j < PER1; ++j) {
                bins[j] = (int)hist[b0 + j];
                own += bins[j];
            }
        }
        int v = own;  // sum over this warp's lanes >= lane
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int t = __shfl_down_sync(0xFFFFFFFFu, v, off);
            if (lane + off < 32) v += t;
        }
        if (lane == 0) wsum[warp] = (uint32_t)v;
        __syncthreads();
        int above = v - own;
        for (int w = warp + 1; w < SELECT_THREADS / 32; ++w) above += (int)wsum[w];
        if (shared) {
            // Thread 0's suffix sum is the slice's total: every block learns it.
            if (tid == 0)
                for (int c = 0; c < C; ++c) st_rank(map_rank(&slice_sum[rank], c), (uint32_t)(above + own));
            cluster_sync_all();
            for (int c = rank + 1; c < C; ++c) above += (int)slice_sum[c];
        }
        if (GROUPED) {
            // Each bin's count becomes, in the first block, the place of its first candidate.
            int place = above;
#pragma unroll
            for (int j = PER1 - 1; j >= 0; --j)
                if (j < per) {
                    if (shared) st_rank(map_rank(&hist[b0 + j], 0), (uint32_t)place);
                    else hist[b0 + j] = (uint32_t)place;
                    place += bins[j];
                }
        }
        if (n > q && above < q && above + own >= q) {  // exactly one thread: the n_l-th best key is in its bins
            int cum = above;
#pragma unroll
            for (int j = PER1 - 1; j >= 0; --j) {
                if (j < per) {
                    const int h = bins[j];
                    if (cum < q && cum + h >= q) {
                        const int coarse = GROUPED ? h <= SEL_BND : cum + h <= sort_cap;
                        const int take = GROUPED || !coarse ? cum : cum + h;  // (narrowed: until then those above)
                        for (int c = 0; c < parts; ++c) {
                            const int to = shared ? c : rank;
                            if (to == rank) {
                                st.code_b = b0 + j;
                                st.n_take = take;
                                st.coarse = coarse;
                            } else {
                                st_rank(map_rank(&st.code_b, to), (uint32_t)(b0 + j));
                                st_rank(map_rank(&st.n_take, to), (uint32_t)take);
                                st_rank(map_rank(&st.coarse, to), (uint32_t)coarse);
                            }
                        }
                    }
                    cum += h;
                }
            }
        }
        if (shared) cluster_sync_all();
        else __syncthreads();
    }

    if (__builtin_expect(!st.coarse, 0)) {  // the same in all blocks
        static_assert(!GROUPED || SEL_BND * sizeof(uint64_t) >= SEL_BINS * sizeof(uint32_t), "room for the counts");
        // Grouped: counted where the bin's candidates go later (the bins keep their places).
        uint32_t* const h2 = GROUPED ? reinterpret_cast<uint32_t*>(bkey) : hist;
        if constexpr (GROUPED)
            narrow_bin_apart<C>(I.ckey, I.cyx, n, parts, q, st.n_take, sort_cap, h2, wsum, tie, st, &s_cnt);
        else
            narrow_bin<C, false>(I.ckey, I.cyx, n, parts, q, st.n_take, sort_cap, h2, wsum, tie, st, &s_cnt);
    }
    auto keep = [&](int pos, uint64_t key, uint32_t yx) {
        I.kkey[pos] = key;
        I.kyx[pos] = yx;
    };
    if constexpr (GROUPED) {
        // Gather: the better bins to their places, the boundary bin to the first block.
        const int code_b = st.code_b;
        const bool split = st.split != 0;
        const ulonglong2* ck2 = reinterpret_cast<const ulonglong2*>(I.ckey);
        const int n2 = (n + 1) >> 1;
        // A place of the first block's counter.
        auto take = [&](void* counter) {
            return shared ? atomic_add_rank(map_rank(counter, 0), 1) : atomicAdd(static_cast<int*>(counter), 1);
        };
        auto bound = [&](uint64_t key, uint32_t yx) {
            const int pos = take(&s_bnd);  // at most SEL_BND of them
            if (pos < SEL_BND) {
                if (shared) {
                    st_rank64(map_rank(&bkey[pos], 0), key);
                    st_rank(map_rank(&byx[pos], 0), yx);
                } else {
                    bkey[pos] = key;
                    byx[pos] = yx;
                }
            }
        };
        if (__builtin_expect(split, 0)) {
            const uint64_t pre_hi = st.pre_hi, msk_hi = st.msk_hi;
            const uint32_t pre_lo = st.pre_lo, msk_lo = st.msk_lo;
            for (int i0 = i_first; i0 < n; i0 += SEL_UNROLL * i_step) {
                uint64_t hi[SEL_UNROLL];
                uint32_t yx[SEL_UNROLL];
#pragma unroll
                for (int k = 0; k < SEL_UNROLL; ++k) {
                    const int i = i0 + k * i_step;
                    hi[k] = i < n ? I.ckey[i] : 0ull;
                    yx[k] = i < n ? I.cyx[i] : 0u;
                }
#pragma unroll
                for (int k = 0; k < SEL_UNROLL; ++k) {
                    const int code = (int)key_code(hi[k]);
                    if (i0 + k * i_step >= n || code < code_b) continue;
                    const uint64_t mh = hi[k] & msk_hi;
                    const uint32_t ml = ~yx[k] & msk_lo;
                    if (code == code_b && rank_less(mh, ml, pre_hi, pre_lo)) continue;
                    if (code == code_b && mh == pre_hi && ml == pre_lo) {
                        bound(hi[k], yx[k]);
                    } else {
                        const int pos = code > code_b ? take(&hist[code]) : take(&s_cnt);
                        if (pos < q) keep(pos, hi[k], yx[k]);
                    }
                }
            }
        }
        for (int i0 = split ? n2 : i_first; i0 < n2; i0 += SEL_UNROLL * i_step) {
            ulonglong2 v[SEL_UNROLL];
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
                if (2 * i + 1 < n) v[k] = ck2[i];
                else v[k] = make_ulonglong2(2 * i < n ? I.ckey[2 * i] : 0ull, 0ull);
            }
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int i = 2 * (i0 + k * i_step) + h;
                    if (i >= n) continue;
                    const uint64_t key = h ? v[k].y : v[k].x;
                    const int code = (int)key_code(key);
                    if (code < code_b) continue;
                    const uint32_t yx = I.cyx[i];
                    if (code > code_b) {
                        const int pos = take(&hist[code]);
                        if (pos < q) keep(pos, key, yx);
                    } else {
                        bound(key, yx);
                    }
                }
            }
        }
        if (shared) cluster_sync_all();
        else __syncthreads();
        if (rank != 0) return;
        // The boundary bin: its best fill the rest, found by the fine codes.
        static_assert(SELECT_THREADS == 512, "one fine code, or digit of a rank word, per thread");
        const int nb = min(s_bnd, SEL_BND), above = st.n_take + st.sure, need = q - above;
        if (nb == 0) {
            if (tid == 0) I.ctr[1] = above;
            return;
        }
        uint16_t* const left = reinterpret_cast<uint16_t*>(hist + 1024);  // boundary candidates
        int base = above, nl = nb;  // the place of the best of them, their number
        if (!split) {
            hist[tid] = 0u;
            if (tid == 0) {
                s_left = 0;
                s_cnt = above;
            }
            __syncthreads();
            for (int i = tid; i < nb; i += SELECT_THREADS) atomicAdd(&hist[fine_bits(bkey[i])], 1u);
            __syncthreads();
            const int own = (int)hist[tid], better = threads_after(own, wsum, tid);
            if (better < need && better + own >= need) s_fine = tid | better << 9;  // exactly one thread
            __syncthreads();
            const int fine = s_fine & 511;
            base += s_fine >> 9;  // candidates above the fine boundary bin
            for (int i = tid; i < nb; i += SELECT_THREADS) {
                const int c = (int)fine_bits(bkey[i]);
                if (c > fine) {
                    const int pos = atomicAdd(&s_cnt, 1);
                    keep(pos, bkey[i], byx[i]);
                } else if (c == fine) {
                    left[atomicAdd(&s_left, 1)] = (uint16_t)i;
                }
            }
            __syncthreads();
            nl = s_left;
        } else {
            for (int i = tid; i < nb; i += SELECT_THREADS) left[i] = (uint16_t)i;
            __syncthreads();
        }
        if (__builtin_expect(nl > SEL_RANK, 0)) {
            rank_ties(bkey, byx, hist, left, nl, base, q, wsum, tie, &s_left, &s_cnt, &s_fine, I.kkey, I.kyx);
            nl = 0;
        }
        for (int i = tid; i < nl; i += SELECT_THREADS) {
            const uint64_t key = bkey[left[i]];
            const uint32_t yx = byx[left[i]];
            int place = base;
            for (int j = 0; j < nl; ++j) place += rank_less(key, ~yx, bkey[left[j]], ~byx[left[j]]);
            if (place < q) keep(place, key, yx);
        }
        if (tid == 0) I.ctr[1] = q;
        return;
    }

    // Gather, each block its part of the candidates: code >= b, or, of a narrowed
    // bin b, those whose masked rank word is >= the prefix.
    const int n_take = st.n_take;
    const uint32_t code_b = (uint32_t)st.code_b;
    auto gather = [&](uint64_t key, uint32_t yx) {
        const int pos = atomicAdd(&s_cnt, 1);
        if (pos < sort_cap) {
            skey[pos] = key;
            syx[pos] = yx;
        }
    };
    if (__builtin_expect(st.split, 0)) {
        const uint64_t pre_hi = st.pre_hi, msk_hi = st.msk_hi;
        const uint32_t pre_lo = st.pre_lo, msk_lo = st.msk_lo;
        for (int i0 = i_first; i0 < n; i0 += SEL_UNROLL * i_step) {
            uint64_t hi[SEL_UNROLL];
            uint32_t yx[SEL_UNROLL];
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
                hi[k] = i < n ? I.ckey[i] : 0ull;
                yx[k] = i < n ? I.cyx[i] : 0u;
            }
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const uint32_t code = key_code(hi[k]);
                if (i0 + k * i_step >= n || code < code_b ||
                    (code == code_b && rank_less(hi[k] & msk_hi, ~yx[k] & msk_lo, pre_hi, pre_lo)))
                    continue;
                gather(hi[k], yx[k]);
            }
        }
    } else {
        const ulonglong2* ck2 = reinterpret_cast<const ulonglong2*>(I.ckey);
        const int n2 = (n + 1) >> 1;
        for (int i0 = i_first; i0 < n2; i0 += SEL_UNROLL * i_step) {
            ulonglong2 v[SEL_UNROLL];
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
                if (i < n2) {
                    if (2 * i + 1 < n) v[k] = ck2[i];
                    else v[k] = make_ulonglong2(I.ckey[2 * i], 0ull);
                } else {
                    v[k] = make_ulonglong2(0ull, 0ull);
                }
            }
#pragma unroll
            for (int k = 0; k < SEL_UNROLL; ++k) {
                const int i = i0 + k * i_step;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint64_t key = h ? v[k].y : v[k].x;
                    if (i < n2 && 2 * i + h < n && key_code(key) >= code_b) gather(key, I.cyx[2 * i + h]);
                }
            }
        }
    }
    if (shared) {
        // The first block's own entries stay in place; the others append theirs.
        cluster_sync_all();
        if (rank != 0) {
            const int cnt = min(s_cnt, sort_cap);
            if (tid == 0) st.at = atomic_add_rank(map_rank(&s_cnt, 0), cnt);
            __syncthreads();
            const int base = st.at;
            for (int i = tid; i < cnt && base + i < sort_cap; i += SELECT_THREADS) {
                st_rank64(map_rank(&skey[base + i], 0), skey[i]);
                st_rank(map_rank(&syx[base + i], 0), syx[i]);
            }
        }
        cluster_sync_all();
        if (rank != 0) return;
    }
    __syncthreads();
    const int got = min(min(s_cnt, n_take), sort_cap);
    int P = SEL_MIN_SORT;
    while (P < got) P <<= 1;
    for (int i = got + tid; i < P; i += SELECT_THREADS) {
        skey[i] = 0ull;           // below every real candidate (keys never reach -2^63)
        syx[i] = 0xFFFFFFFFu;
    }
    __syncthreads();
    bitonic_sort(skey, syx, P, tid);
    const int out = min(got, m);
    for (int i = tid; i < out; i += SELECT_THREADS) {
        I.kkey[i] = skey[i];
        I.kyx[i] = syx[i];
    }
    if (tid == 0) I.ctr[1] = out;
}

// Sort-buffer entries: room for twice the largest quota (the coarse pass's
// boundary bin), else the quota rounded up to a power of two; at least
// SEL_MIN_SORT.
static int select_sort_cap(int max_quota) {
    int P = SEL_MIN_SORT / 2;
    while (P < max_quota) P <<= 1;
    return 2 * P * (int)(sizeof(uint64_t) + sizeof(uint32_t)) <= SEL_MAX_DYN ? 2 * P : P;
}

int select_smem_bytes(int max_quota) {
    return select_sort_cap(max_quota) * (int)(sizeof(uint64_t) + sizeof(uint32_t));
}

// The orientation kernel's ranking costs each keypoint a sixth more where few keys
// share a code, and the length of its run where many do (a smooth scene): with n_l
// keypoints over a fixed number of codes, n_l^2 an image, 0.75 us per million.  The
// sort is one block's chain of barriers, which the images of a launch share: 6 us
// for 1000 keypoints, 15 for 2000, 55 for 4096, 150 for 8192, so at least three
// times the largest image's ranking.  Lists stay grouped while the images' n_l^2 add
// up to at most four times the largest's (a frame of 8 levels counts 1.9), or to no
// more than a short sort costs.  Whole calls, grouped / sorted, us: two 1080p levels
// of 8192 features 123 / 239, two 1080p frames of 8 levels and 8192 137 / 156, and
// 1000 114 / 117; 8 720p levels of 1000 83 / 95, of 4096 227 / 163, of 8192 516 / 284;
// 16 of 8192 986 / 378; 32 of 1000 232 / 211, of 8192 1876 / 538 (sorted by one block
// an image, without the fused stages: 351, 246, 193; 157, 235, 385; 480; 281, 670).
bool select_grouped(int n_img, int64_t quota_sq, int max_quota) {
    return n_img <= 32 && quota_sq <= std::max<int64_t>(4ll * max_quota * max_quota, 16000000);
}

template <int C, bool GROUPED>
static void launch_select_t(const Img* imgs, int n_img, int levels, const Call* call, int mq, cudaStream_t st,
                            bool pdl) {
    launch_chain(k_select<C, GROUPED>, dim3(n_img / levels * C, levels), SELECT_THREADS,
                 GROUPED ? 0 : select_smem_bytes(mq), st, pdl, C, imgs, call, GROUPED ? 0 : select_sort_cap(mq));
}

// Blocks per image, by the images of the launch.  A cluster shortens the scan
// of the largest image, which sets the launch's length, until its blocks no
// longer fit the chip beside each other (four 512-thread blocks on each of
// 152 SMs): 8 while every image has SMs of its own (grouped lists of up to 16
// images; sorted ones are better with 4: 16 VGA frames of 4096, whole call 240
// against 216 us), 4 up to 128 images, 2 up to 304.  Measured stage times of sorted lists (1080p, 8 levels; 1 / 2 / 4 / 8
// blocks): 8 images 41 / 33 / 27 / 22 us, 32 images 43 / 35 / 26 / 28, 128
// images 49 / 39 / 35 / 41, 304 images 64 / 57 / 64 / 84, 1024 images 97 / 119
// / 149 / 218.
// Order of the images: with more of them than the chip holds beside each other
// (C <= 2), level by level over the frames, so that the large images start first
// and the small ones fill the SMs after them: 32 frames (256 images) 42 -> 37 us,
// 128 frames 82 -> 60 (whole calls 827 -> 822, 2943 -> 2921).  With clusters of
// 4 they all start at once, and frame by frame is the better one (6 frames, whole
// call: 214 against 216 us).
void launch_select(const Img* imgs, int n_img, int levels, const Call* call, int max_quota, bool grouped, void* stream,
                   bool pdl) {
    if (n_img <= 0) return;
    const int mq = max_quota > 0 ? max_quota : 1;
    const cudaStream_t st = (cudaStream_t)stream;
    // Sorted lists of large quotas: no more blocks than are resident at once, by their shared
    // memory (whole calls of 40 VGA levels of 4096 features: 352 us with four blocks each, 286
    // with two; of 96 720p levels of 8192: 1351 and 1167).
    const int per_sm = std::min(4, (227 * 1024) / (select_smem_bytes(mq) + 18 * 1024)), fit = 152 * std::max(per_sm, 1);
    if (grouped && n_img <= 16) launch_select_t<8, true>(imgs, n_img, 1, call, mq, st, pdl);
    else if (grouped) launch_select_t<4, true>(imgs, n_img, 1, call, mq, st, pdl);
    else if (n_img <= 128 && 4 * n_img <= fit) launch_select_t<4, false>(imgs, n_img, 1, call, mq, st, pdl);
    else if (n_img <= 304 && 2 * n_img <= fit) launch_select_t<2, false>(imgs, n_img, levels, call, mq, st, pdl);
    else launch_select_t<1, false>(imgs, n_img, levels, call, mq, st, pdl);
}

// The limit is a per-device attribute of the kernel shared by every handle,
// server slot and allocation-free call, so it only ever grows: a later caller
// with a smaller quota must not lower it under an earlier one.
void set_select_smem_limit(int bytes) {
    static std::mutex mu;
    static int limit[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && bytes <= limit[dev]) return;
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const bool ok = cudaFuncSetAttribute(k_select<1, false>, attr, bytes) == cudaSuccess &&
                    cudaFuncSetAttribute(k_select<2, false>, attr, bytes) == cudaSuccess &&
                    cudaFuncSetAttribute(k_select<4, false>, attr, bytes) == cudaSuccess;
    if (ok && dev >= 0 && dev < 64) limit[dev] = bytes;
}

}  // namespace ofk
