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

static PyrAxis pyramid_ranges(const int32_t* sizes, const int32_t* const* tab, int nl, int nt, int max_extent, bool columns) {
    PyrAxis A;
    A.nt = nt;
    A.nl = nl;
    // Tile boundaries: equal shares of every level, columns at multiples of 4.
    auto bound = [&](int l, int i) {
        if (i >= nt) return sizes[l];
        const int b = (int)((int64_t)sizes[l] * i / nt);
        return columns ? b & ~3 : b;
    };
    A.ranges.assign((size_t)nt * (nl + 1), PyrRange());
    A.extent.assign(nl + 1, 0);
    int words = 0;
    for (int i = 0; i < nt; ++i) {
        PyrRange* const tile = A.ranges.data() + (size_t)i * (nl + 1);
        int n = 4 * (nl + 1);
        for (int l = nl; l >= 0; --l) {
            PyrRange& R = tile[l];
            int n0 = 0, n1 = 0;  // needed: the owned range and the sources of the next level's computed range
            if (l > 0) {
                R.o0 = n0 = bound(l, i);
                R.o1 = n1 = std::max(bound(l, i + 1), R.o0);
            }
            if (l < nl && tile[l + 1].c1 > tile[l + 1].c0) {
                const PyrRange& N = tile[l + 1];
                const int d1 = std::min(N.c1, sizes[l + 1]) - 1;
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
    A.ok = A.extent[0] <= max_extent;
    A.stride = (words + 3) / 4 * 4;
    return A;
}

static void pyramid_blocks(const PyrAxis& A, const int32_t* sizes, const int32_t* const* tab, const int32_t* row_words,
                    int32_t* out) {
    const bool columns = row_words == nullptr;
    const int nl = A.nl;
    for (int i = 0; i < A.nt; ++i) {
        const PyrRange* const tile = A.ranges.data() + (size_t)i * (nl + 1);
        int32_t* b = out + (size_t)A.stride * i;
        int32_t* e = b + 4 * (nl + 1);
        for (int l = 0; l <= nl; ++l) {
            const PyrRange& R = tile[l];
            b[4 * l] = R.c0;
            b[4 * l + 1] = !columns ? (R.c1 - R.c0) | row_words[l] << 16 : l > 0 ? pack_groups((R.c1 - R.c0) / 4) : R.c1 - R.c0;
            b[4 * l + 2] = R.o0;
            b[4 * l + 3] = R.o1;
            if (l == 0) continue;
            const int s0 = tile[l - 1].c0;
            const int32_t* const tl = tab[l];
            if (!columns) {
                const int rw = row_words[l - 1];
                for (int d = R.c0; d < R.c1; ++d) {
                    const int t = tl[d];
                    *e++ = (int32_t)((uint32_t)(((t >> 12) - s0) * rw) << 16) | 2 * (t & 4095);
                }
                continue;
            }
            auto weights = [](int t) { return (int32_t)(4096u + 2u * (uint32_t)(t & 4095) * 0xFFFFu); };  // 4096 - 2a | 2a << 16
            auto pair = [](int o) { return (uint32_t)(o | (o + 1) << 4); };  // selects bytes o, o + 1
            const int last = sizes[l] - 1;
            for (int d = R.c0; d < R.c1; d += 4, e += 8) {
                const int t0 = tl[std::min(d, last)], t1 = tl[std::min(d + 1, last)], t2 = tl[std::min(d + 2, last)],
                          t3 = tl[std::min(d + 3, last)];
                const int x0 = (t0 >> 12) - s0, x1 = (t1 >> 12) - s0, x2 = (t2 >> 12) - s0, x3 = (t3 >> 12) - s0;
                const int wa = x0 >> 2, wb = x2 >> 2;
                e[0] = wa | (wb << 16);
                e[1] = (int32_t)(pair(x0 - 4 * wa) | pair(x1 - 4 * wa) << 8 | pair(x2 - 4 * wb) << 16 | pair(x3 - 4 * wb) << 24);
                e[2] = weights(t0);
                e[3] = weights(t1);
                e[4] = weights(t2);
                e[5] = weights(t3);
            }
        }
    }
}

bool pyramid_pieces(const std::vector<int32_t>& ws, const std::vector<int32_t>& hs, const std::vector<const int32_t*>& xtab,
                    const std::vector<const int32_t*>& ytab, int max_levels, int tile, double max_seam,
                    std::vector<PyrPiece>& out) {
    const int nl = (int)ws.size();
    // Levels whose source columns step by at most 3 (the kernel picks byte pairs of 4 outputs from two
    // words): a step is at most the ratio of the widths, rounded up.
    std::vector<char> steps(nl, 1);
    for (int l = 1; l < nl; ++l)
        if (10 * (int64_t)ws[l - 1] > 29 * (int64_t)ws[l])
            for (int d = 1; d < ws[l] && steps[l]; ++d) steps[l] = (xtab[l][d] >> 12) - (xtab[l][d - 1] >> 12) <= 3;
    for (int a = 0; a + 1 < nl;) {
        int most = 0;
        while (a + 1 + most < nl && most < max_levels && steps[a + 1 + most]) ++most;
        bool found = false;
        for (int t = tile; t >= 32 && !found; t = t > 128 ? 128 : t / 2)
            for (int n = most; n >= 1 && !found; --n) {
                PyrPiece p;
                p.level = a;
                p.nl = n;
                p.ntx = (ws[a] + t - 1) / t;
                p.nty = (hs[a] + t - 1) / t;
                p.x = pyramid_ranges(ws.data() + a, xtab.data() + a, n, p.ntx, 256, true);
                // (A seam is at least its columns' part.)
                if (!p.x.ok || (n > 1 && (double)p.x.computed > max_seam * (double)p.x.owned)) continue;
                p.y = pyramid_ranges(hs.data() + a, ytab.data() + a, n, p.nty, 256, false);
                if (!p.y.ok) continue;
                const double seam = (double)p.x.computed * p.y.computed / ((double)p.x.owned * p.y.owned);
                if (n > 1 && seam > max_seam) continue;
                out.push_back(std::move(p));
                a += n;
                found = true;
            }
        if (!found) return false;
    }
    return true;
}

void pyramid_tables(const PyrPiece& p, const std::vector<int32_t>& ws, const std::vector<int32_t>& hs,
                    const std::vector<const int32_t*>& xtab, const std::vector<const int32_t*>& ytab, int32_t* x, int32_t* y) {
    std::vector<int32_t> row_words(p.nl + 1);
    for (int l = 0; l <= p.nl; ++l) row_words[l] = std::max(p.x.extent[l], 16) / 4;
    pyramid_blocks(p.x, ws.data() + p.level, xtab.data() + p.level, nullptr, x);
    pyramid_blocks(p.y, hs.data() + p.level, ytab.data() + p.level, row_words.data(), y);
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
