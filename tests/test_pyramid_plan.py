"""Host planning of the fused pyramid (csrc/of_plan.cpp), compiled with a small program.

Runs and tables: every pixel of every level is owned by one tile; what a tile computes covers what
it owns and what its later levels read; weights, byte pairs and row offsets give each output's
source samples.  Cost: planning is part of the first call with a shape, so it may take no more
than a small multiple of making the resize tables that it starts from."""

import os
import subprocess
import sys

import pytest

import paper_2506_07164_gb300 as ofg

b = sys.modules[ofg.build.__module__]  # the build module (the package exports its function under the same name)

PROGRAM = r"""
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include "of_plan.h"
using namespace ofh;
struct Levels {
    std::vector<int32_t> ws, hs;
    std::vector<std::vector<int32_t>> x, y;
    std::vector<const int32_t*> xt, yt;
    Levels(int w, int h, int nl, float scale) : ws(nl), hs(nl) {
        level_sizes(w, h, nl, scale, ws.data(), hs.data(), nullptr);
        int k = 0;
        while (k < nl && ws[k] > 0 && hs[k] > 0) ++k;
        ws.resize(k), hs.resize(k);
    }
    void tables() {
        const size_t k = ws.size();
        x.resize(k), y.resize(k), xt.assign(k, nullptr), yt.assign(k, nullptr);
        for (size_t l = 1; l < k; ++l) {
            x[l].resize(ws[l]), y[l].resize(hs[l]);
            resize_table(ws[l - 1], ws[l], x[l].data());
            resize_table(hs[l - 1], hs[l], y[l].data());
            xt[l] = x[l].data(), yt[l] = y[l].data();
        }
    }
};
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s (%dx%d tile %d)\n", __LINE__, #c, L.ws[0], L.hs[0], tile); return 1; } } while (0)
static int check(Levels& L, int tile, double seam) {
    std::vector<PyrPiece> ps;
    L.tables();
    if (!pyramid_pieces(L.ws, L.hs, L.xt, L.yt, 15, tile, seam, ps)) return -1;
    int level = 0;
    for (const PyrPiece& p : ps) {
        CHECK(p.level == level && p.nl >= 1 && p.nl <= 15);
        level += p.nl;
        std::vector<int32_t> bx((size_t)p.x.stride * p.x.nt, 0), by((size_t)p.y.stride * p.y.nt, 0);
        pyramid_tables(p, L.ws, L.hs, L.xt, L.yt, bx.data(), by.data());
        for (int axis = 0; axis < 2; ++axis) {
            const PyrAxis& A = axis ? p.y : p.x;
            const std::vector<int32_t>& size = axis ? L.hs : L.ws;
            const auto& tab = axis ? L.yt : L.xt;
            std::vector<int> next(p.nl + 1, 0);
            for (int i = 0; i < A.nt; ++i) {
                const int32_t* h = (axis ? by : bx).data() + (size_t)A.stride * i;
                const int32_t* e = h + 4 * (p.nl + 1);
                int s0 = h[0], s1 = h[0] + (axis ? h[1] & 0xFFFF : h[1]);
                CHECK(axis || s0 % 16 == 0);
                CHECK(s1 - s0 <= 256 && s1 - s0 <= A.extent[0]);
                for (int l = 1; l <= p.nl; ++l) {
                    const int32_t* q = h + 4 * l;
                    const int n = size[p.level + l], groups = q[1] & 255;
                    const int c0 = q[0], c1 = c0 + (axis ? q[1] & 0xFFFF : 4 * groups);
                    const int rw = axis ? (h[4 * (l - 1) + 1] >> 16) : 0;
                    CHECK(q[2] == next[l] && q[3] >= q[2]);
                    next[l] = q[3];
                    CHECK(q[2] == q[3] || (c0 <= q[2] && q[3] <= c1));
                    CHECK(c1 - c0 <= A.extent[l]);
                    if (axis) {
                        for (int d = c0; d < c1; ++d) {
                            const int t = tab[p.level + l][d], src = t >> 12, a2 = 2 * (t & 4095);
                            const uint32_t v = (uint32_t)*e++;
                            CHECK((int)(v & 0xFFFF) == a2 && (int)(v >> 16) == (src - s0) * rw);
                            CHECK(src >= s0 && (a2 == 0 ? src : src + 1) < s1);
                        }
                    } else {
                        CHECK(c0 % 4 == 0 && groups <= 64 && (groups == 0 || (q[1] >> 8) == (65536 + groups - 1) / groups));
                        for (int d = c0; d < c1; d += 4, e += 8)
                            for (int k = 0; k < 4; ++k) {
                                const int t = tab[p.level + l][std::min(d + k, n - 1)], a2 = 2 * (t & 4095);
                                const uint32_t w = (uint32_t)e[2 + k], word = k < 2 ? (uint32_t)e[0] & 0xFFFF : (uint32_t)e[0] >> 16;
                                const uint32_t sel = (uint32_t)e[1] >> (8 * k) & 0xFF;
                                CHECK(w == ((4096u - a2) | (uint32_t)a2 << 16));
                                const int lo = 4 * word + (sel & 7), hi = 4 * word + (sel >> 4 & 7);
                                CHECK((sel & 0x88) == 0 && lo == (t >> 12) - s0 && hi == lo + 1);
                                CHECK((t >> 12) >= s0 && (a2 == 0 ? t >> 12 : (t >> 12) + 1) < s1);
                            }
                    }
                    s0 = c0, s1 = c1;
                }
            }
            for (int l = 1; l <= p.nl; ++l) CHECK(next[l] == size[p.level + l]);
        }
    }
    CHECK(level == (int)L.ws.size() - 1);
    return 0;
}
int main(int, char** a) {
    using C = std::chrono::steady_clock;
    if (a[1][0] == 'c') {
        std::srand(std::atoi(a[2]));
        int done = 0;
        for (int i = 0; i < 300; ++i) {
            const int w = 1 + std::rand() % (i % 3 ? 2000 : 200), h = 1 + std::rand() % (i % 5 ? 1500 : 100);
            Levels L(w, h, 2 + std::rand() % 15, 1.01f + (float)(std::rand() % 1000) / 1000.f * (i % 4 ? 0.6f : 2.9f));
            const int tile[4] = {64, 96, 128, 160}, k = std::rand() % 4;
            const int rc = check(L, tile[k], k == 3 ? 1.06 : 1.9);
            if (rc > 0) return 1;
            done += rc == 0;
        }
        std::printf("%d\n", done);
        return 0;
    }
    double tables = 1e30, plan = 1e30;
    for (int rep = 0; rep < 5; ++rep) {
        double t = 0, p = 0;
        for (int f = 0; f < 64; ++f) {
            Levels L(640 + 18 * f, 480 + 8 * f, 8, 1.2f);
            const auto t0 = C::now();
            L.tables();
            const auto t1 = C::now();
            std::vector<PyrPiece> ps;
            if (!pyramid_pieces(L.ws, L.hs, L.xt, L.yt, 15, 160, 1.06, ps)) return 1;
            for (const PyrPiece& q : ps) {
                std::vector<int32_t> x((size_t)q.x.stride * q.x.nt, 0), y((size_t)q.y.stride * q.y.nt, 0);
                pyramid_tables(q, L.ws, L.hs, L.xt, L.yt, x.data(), y.data());
            }
            const auto t2 = C::now();
            t += std::chrono::duration<double>(t1 - t0).count();
            p += std::chrono::duration<double>(t2 - t1).count();
        }
        tables = std::min(tables, t), plan = std::min(plan, p);
    }
    std::printf("%.3f\n", plan / tables);
}
"""


@pytest.fixture(scope="module")
def planner(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "planner.cpp").write_text(PROGRAM)
    exe = str(d / "planner")
    r = subprocess.run(["g++", *b.CXX_FLAGS, str(d / "planner.cpp"), os.path.join(b.CSRC, "of_plan.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_runs_and_tables(planner, seed):
    r = subprocess.run([planner, "c", str(seed)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 200


def test_planning_costs_no_more_than_a_few_tables(planner):
    """64 frame sizes at 8 levels, in short runs (what large batches take): 7 times the resize tables when
    every try of the search made tables and blocks of its own, about half of them with the search on ranges."""
    r = subprocess.run([planner, "t"], capture_output=True, text=True)
    assert r.returncode == 0
    assert float(r.stdout) < 4.0, r.stdout
