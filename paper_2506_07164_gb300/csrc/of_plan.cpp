// Host-side plan arithmetic: pyramid level sizes, per-level feature quotas,
// bilinear source-coordinate tables and the exact fraction for Harris k.
// Compiled with -ffp-contract=off: every float64 step below is one IEEE
// operation, so the tables are identical on every host.
#include <math.h>
#include <stdint.h>

#include "of_plan.h"

#include <algorithm>

namespace ofh {

// Level l has scale s_l = scale^l, a float64 running product starting at 1;
// w_l = floor(W / s_l + 0.5), h_l likewise (Sec. 1; Sec. 6.1 "decrease exponentially").
void level_sizes(int W, int H, int levels, float scale, int32_t* ws, int32_t* hs, double* ls) {
    double s = 1.0;
    for (int l = 0; l < levels; ++l) {
        ws[l] = (l == 0) ? W : (int32_t)floor((double)W / s + 0.5);
        hs[l] = (l == 0) ? H : (int32_t)floor((double)H / s + 0.5);
        if (ls) ls[l] = s;
        s = s * (double)scale;
    }
}

// Quota of level l for N features: proportional to level area, ratio
// f = 1/scale^2 per level: round(N (1-f)/(1-f^L) f^l), capped by what is left;
// the last level takes the remainder.
void level_quotas(int N, int L, float scale, int32_t* q) {
    const double sc = (double)scale;
    const double f = 1.0 / (sc * sc);
    double fpow = 1.0;
    for (int l = 0; l < L; ++l) fpow = fpow * f;
    const double share = (1.0 - f) / (1.0 - fpow);
    int left = N;
    double fl = 1.0;
    for (int l = 0; l < L; ++l) {
        int n;
        if (l + 1 == L) {
            n = left;
        } else {
            n = (int)floor((double)N * share * fl + 0.5);
            if (n > left) n = left;
        }
        q[l] = n;
        left -= n;
        fl = fl * f;
    }
}

// Source sample of each of n_dst destination pixels for a centre-aligned
// bilinear resize from n_src pixels: s = (d + 0.5) * (n_src / n_dst) - 0.5,
// clamped to [0, n_src - 1]; entry = (floor(s) << 12) | lrint(frac(s) * 2048).
void resize_table(int n_src, int n_dst, int32_t* tab) {
    const double ratio = (double)n_src / (double)n_dst;
    const double last = (double)(n_src - 1);
    for (int d = 0; d < n_dst; ++d) {
        double s = ((double)d + 0.5) * ratio - 0.5;
        s = s < 0.0 ? 0.0 : (s > last ? last : s);
        const double i0 = floor(s);
        const int32_t a = (int32_t)lrint((s - i0) * 2048.0);
        tab[d] = ((int32_t)i0 << 12) | a;
    }
}

// Harris k rounded to a multiple of 1e-6 and reduced to num/den.  The integer
// key den*det - num*trace^2 fits int64 for 7x7 windows when 0 <= k <= 0.25
// and den <= 3000; anything else is rejected.
bool k_fraction(float k, int64_t* num, int64_t* den) {
    const double kd = (double)k;
    if (!(kd >= 0.0 && kd <= 0.25)) return false;
    int64_t n = (int64_t)llrint(kd * 1000000.0), d = 1000000;
    int64_t a = n, b = d;
    while (b != 0) {
        const int64_t r = a % b;
        a = b;
        b = r;
    }
    if (a == 0) a = d;
    n /= a;
    d /= a;
    if (d > 3000) return false;
    *num = n;
    *den = d;
    return true;
}

// A level's column groups n (at most 64) and ceil(2^16 / n), which divides thread numbers by n: n | m << 8.
static int32_t pack_groups(int n) { return n > 0 ? n | ((65536 + n - 1) / n << 8) : 0; }

PyrAxis pyramid_axis(const int32_t* sizes, int nl, int nt, int max_extent, const int32_t* row_words) {
    const bool columns = row_words == nullptr;
    PyrAxis A;
    A.nt = nt;
    A.nl = nl;
    A.ok = true;
    std::vector<std::vector<int32_t>> tab(nl + 1);
    for (int l = 1; l <= nl; ++l) {
        tab[l].resize(sizes[l]);
        resize_table(sizes[l - 1], sizes[l], tab[l].data());
        if (columns)
            for (int d = 1; d < sizes[l]; ++d)
                if ((tab[l][d] >> 12) - (tab[l][d - 1] >> 12) > 3) A.ok = false;
    }
    // Tile boundaries: equal shares of every level, columns at multiples of 4.
    auto bound = [&](int l, int i) {
        if (i >= nt) return sizes[l];
        const int b = (int)((int64_t)sizes[l] * i / nt);
        return columns ? b & ~3 : b;
    };
    struct Range {
        int c0 = 0, c1 = 0, o0 = 0, o1 = 0;
    };
    std::vector<std::vector<Range>> tiles(nt, std::vector<Range>(nl + 1));
    A.extent.assign(nl + 1, 0);
    int words = 0;
    for (int i = 0; i < nt; ++i) {
        int n = 4 * (nl + 1);
        for (int l = nl; l >= 0; --l) {
            Range& R = tiles[i][l];
            int n0 = 0, n1 = 0;  // needed: the owned range and the sources of the next level's computed range
            if (l > 0) {
                R.o0 = n0 = bound(l, i);
                R.o1 = n1 = std::max(bound(l, i + 1), R.o0);
            }
            if (l < nl && tiles[i][l + 1].c1 > tiles[i][l + 1].c0) {
                const Range& N = tiles[i][l + 1];
                const int d1 = std::min(N.c1, (int)sizes[l + 1]) - 1;
                const int s0 = tab[l + 1][N.c0] >> 12, s1 = std::min((tab[l + 1][d1] >> 12) + 1, sizes[l] - 1) + 1;
                if (n1 > n0) {
                    n0 = std::min(n0, s0);
                    n1 = std::max(n1, s1);
                } else {
                    n0 = s0;
                    n1 = s1;
                }
            }
            if (n1 > n0) {
                const int q = !columns ? 1 : l > 0 ? 4 : 16;
                R.c0 = n0 / q * q;
                R.c1 = (n1 + q - 1) / q * q;
            }
            A.extent[l] = std::max(A.extent[l], R.c1 - R.c0);
            if (l > 0) {
                n += columns ? (R.c1 - R.c0) / 4 * 8 : R.c1 - R.c0;
                A.computed += R.c1 - R.c0;
                A.owned += R.o1 - R.o0;
            }
        }
        words = std::max(words, n);
    }
    if (A.extent[0] > max_extent) A.ok = false;
    A.stride = (words + 3) / 4 * 4;
    A.blk.assign((size_t)A.stride * nt, 0);
    if (!A.ok) return A;
    for (int i = 0; i < nt; ++i) {
        int32_t* b = A.blk.data() + (size_t)A.stride * i;
        int32_t* e = b + 4 * (nl + 1);
        for (int l = 0; l <= nl; ++l) {
            const Range& R = tiles[i][l];
            b[4 * l] = R.c0;
            b[4 * l + 1] = !columns ? (R.c1 - R.c0) | row_words[l] << 16 : l > 0 ? pack_groups((R.c1 - R.c0) / 4) : R.c1 - R.c0;
            b[4 * l + 2] = R.o0;
            b[4 * l + 3] = R.o1;
            if (l == 0) continue;
            const int s0 = tiles[i][l - 1].c0;
            if (!columns) {
                for (int d = R.c0; d < R.c1; ++d) {
                    const int t = tab[l][d];
                    *e++ = (int32_t)((uint32_t)(((t >> 12) - s0) * row_words[l - 1]) << 16) | 2 * (t & 4095);
                }
                continue;
            }
            for (int d = R.c0; d < R.c1; d += 4) {
                int xo[4];
                uint32_t wgt[4], sel[4];
                for (int k = 0; k < 4; ++k) {
                    const int t = tab[l][std::min(d + k, sizes[l] - 1)];
                    const uint32_t a2 = 2u * (uint32_t)(t & 4095);
                    xo[k] = (t >> 12) - s0;
                    wgt[k] = (4096u - a2) | (a2 << 16);
                }
                const int wa = xo[0] >> 2, wb = xo[2] >> 2;
                for (int k = 0; k < 4; ++k) {
                    const uint32_t o = (uint32_t)(xo[k] - 4 * (k < 2 ? wa : wb));
                    sel[k] = o | ((o + 1u) << 4);
                }
                e[0] = wa | (wb << 16);
                e[1] = (int32_t)(sel[0] | (sel[1] << 8) | (sel[2] << 16) | (sel[3] << 24));
                for (int k = 0; k < 4; ++k) e[2 + k] = (int32_t)wgt[k];
                e += 8;
            }
        }
    }
    return A;
}

float response_scale(int64_t den) {
    const double f = 1.0 / (4.0 * 7.0 * 255.0);
    return (float)((f * f * f * f) / (double)den);
}

}  // namespace ofh

extern "C" int of_plan_levels(int W, int H, int levels, float scale, int n_features, int32_t* ws,
                              int32_t* hs, int32_t* quota) {
    if (W <= 0 || H <= 0 || levels < 1 || levels > 64 || !(scale > 1.0f) || n_features < 0 ||
        !ws || !hs || !quota)
        return -1;
    ofh::level_sizes(W, H, levels, scale, ws, hs, nullptr);
    ofh::level_quotas(n_features, levels, scale, quota);
    return 0;
}
