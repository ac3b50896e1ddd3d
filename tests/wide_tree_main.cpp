// The four-wide form of the host-built BVH on the CPU: its structure (every triangle in exactly one
// leaf, every wide node referenced once, references in range), and its walk, step for step as the
// kernels make it (csrc/wide.cuh), against the walk of the hit/miss links: the same triangle and t,
// a stack that stays within its bound, and an end (tests/test_wide_tree.py compiles this).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "gsp_internal.h"

static int32_t as_int(float f) { int32_t i; std::memcpy(&i, &f, 4); return i; }
static float as_float(int32_t i) { float f; std::memcpy(&f, &i, 4); return f; }

#define CHECK(x)                                                       \
    do {                                                               \
        if (!(x)) {                                                    \
            std::fprintf(stderr, "FAILED (%d triangles): %s\n", nt, #x); \
            return 1;                                                  \
        }                                                              \
    } while (0)

static const int32_t kNone = INT32_MIN, kMiss = 0x7fffffff;

static int check(const std::vector<float>& v, const std::vector<int32_t>& t, int nr, float tmin) {
    const int nt = (int)t.size() / 3;
    HostBVH b;
    CHECK(bvh_build_host(v.data(), (int64_t)v.size() / 3, t.data(), nt, gsp_bvh_params{16, 4, 7, 6}, b).empty());
    const int64_t nw = b.nwide;
    std::vector<float4> wide((size_t)nw * 8);
    for (int64_t i = 0; i < (int64_t)b.wide_of.size(); ++i)
        if (b.wide_of[i] >= 0) gsp_wide_entry(b.bin.data(), i, [&](int32_t j) { return b.wide_of[j]; }, &wide[8 * b.wide_of[i]]);
    if (b.nnodes == 1) {
        CHECK(nw == 0);
        return 0;
    }
    const float* W = (const float*)wide.data();
    std::vector<int> tri_seen(nt, 0), node_seen(nw, 0);
    node_seen[0] = 1;
    for (int64_t i = 0; i < nw; ++i)
        for (int c = 0; c < 4; ++c) {
            const int32_t r = as_int(W[32 * i + 24 + c]);
            if (r == kNone) {
                CHECK(c >= 2);
            } else if (r >= 0) {
                CHECK(r > 0 && r < nw);
                ++node_seen[r];
            } else {
                for (int k = 0; k < (~r & 7); ++k) {
                    CHECK((~r >> 3) + k < nt);
                    ++tri_seen[(~r >> 3) + k];
                }
            }
        }
    for (int s : tri_seen) CHECK(s == 1);
    for (int s : node_seen) CHECK(s == 1);
    std::mt19937 g(nt);
    std::uniform_real_distribution<float> u(-2.0f, 2.0f);
    std::vector<float> R(8 * (size_t)nr);
    for (int i = 0; i < nr; ++i) {
        float* r = &R[8 * (size_t)i];
        for (int k = 0; k < 3; ++k) {
            r[k] = u(g);
            r[4 + k] = u(g);
        }
        if (i % 7 == 0) r[4] = 0.0f;  // axis-parallel directions
        if (i % 13 == 0) r[4] = r[5] = 0.0f;
        if (i % 17 == 0) r[5] = 1e-31f;
        if (i == 18) r[4] = NAN;
        if (i == 19) r[0] = NAN;
        r[3] = i % 5 ? 0.0f : tmin;
        r[7] = i % 3 ? INFINITY : 2.0f;
    }
    std::vector<int32_t> tri(nr);
    std::vector<float> tt(nr);
    bvh_host_walk(b, R.data(), nr, tri.data(), tt.data(), nullptr, nullptr);
    for (int i = 0; i < nr; ++i) {
        const float *r = &R[8 * (size_t)i], *d = r + 4;
        float inv[3], tb = r[7];
        for (int k = 0; k < 3; ++k) inv[k] = 1.0f / (std::fabs(d[k]) < 1e-30f ? std::copysign(1e-30f, d[k]) : d[k]);
        const float pad = std::fmax(-r[3], 0.0f) * 0x1p-18f;
        int32_t best = -1, cur = 0;
        int sp = 0;
        int64_t steps = 0;
        struct { int32_t key, ref; } stk[64];
        const auto pop = [&] {
            while (sp > 0) {
                --sp;
                if (stk[sp].key < 0 || as_float(stk[sp].key & ~3) <= tb) return stk[sp].ref;
            }
            return kNone;
        };
        while (cur != kNone) {
            CHECK(++steps <= nw + nt);
            if (cur >= 0) {
                const float* q = W + 32 * (int64_t)cur;
                int32_t key[4], near_key = kMiss;
                for (int c = 0; c < 4; ++c) {
                    float tn = r[3], tf = INFINITY;
                    for (int k = 0; k < 3; ++k) {
                        const float tc = (q[8 * k + c] - r[k]) * inv[k], h = q[8 * k + 4 + c], a = std::fabs(inv[k]);
                        tn = std::fmax(tn, std::fmaf(-h, a, tc));
                        tf = std::fmin(tf, std::fmaf(h, a, tc));
                    }
                    key[c] = tn <= std::fmaf(std::fmin(tb, tf), 1.0f + 0x1p-19f, pad) ? ((as_int(tn) & ~3) | c) : kMiss;
                    near_key = std::min(near_key, key[c]);
                }
                if (near_key == kMiss) {
                    cur = pop();
                    continue;
                }
                for (int c = 0; c < 4; ++c)
                    if (key[c] != kMiss && key[c] != near_key) {
                        CHECK(sp < 64);
                        stk[sp].key = key[c];
                        stk[sp++].ref = as_int(q[24 + c]);
                    }
                cur = as_int(q[24 + (near_key & 3)]);
                continue;
            }
            for (int k = 0; k < (~cur & 7); ++k) {
                const float* P = (const float*)&b.tris[3 * ((~cur >> 3) + k)];
                float e1[3], e2[3], s[3];
                for (int a = 0; a < 3; ++a) {
                    e1[a] = P[4 + a] - P[a];
                    e2[a] = P[8 + a] - P[a];
                    s[a] = r[a] - P[a];
                }
                const float px = d[1] * e2[2] - d[2] * e2[1], py = d[2] * e2[0] - d[0] * e2[2], pz = d[0] * e2[1] - d[1] * e2[0];
                const float det = e1[0] * px + e1[1] * py + e1[2] * pz;
                if (det == 0) continue;
                const float f = 1.0f / det, uu = f * (s[0] * px + s[1] * py + s[2] * pz);
                const float qx = s[1] * e1[2] - s[2] * e1[1], qy = s[2] * e1[0] - s[0] * e1[2], qz = s[0] * e1[1] - s[1] * e1[0];
                const float vv = f * (d[0] * qx + d[1] * qy + d[2] * qz), th = f * (e2[0] * qx + e2[1] * qy + e2[2] * qz);
                const int32_t id = as_int(P[3]);
                if (uu >= 0 && vv >= 0 && uu + vv <= 1 && th > r[3] && (th < tb || (th == tb && best >= 0 && id < best))) {
                    tb = th;
                    best = id;
                }
            }
            cur = pop();
        }
        CHECK(best == tri[i]);
        CHECK(best < 0 || tb == tt[i]);
    }
    return 0;
}

int main() {
    int bad = 0;
    std::mt19937 g(1);
    std::uniform_real_distribution<float> u(-1.0f, 1.0f);
    for (int nt : {1, 4, 5, 6, 7, 8, 9, 17, 36, 100, 1000, 20000}) {
        std::vector<float> v;
        std::vector<int32_t> t;
        for (int i = 0; i < 3 * nt; ++i) t.push_back(i);
        for (int i = 0; i < nt; ++i) {
            const float c[3] = {u(g), u(g), u(g)};
            for (int k = 0; k < 9; ++k) v.push_back(c[k % 3] + 0.2f * u(g));
        }
        bad += check(v, t, 4000, -3.0f);
    }
    {  // a flat grid: boxes without extent along one axis
        std::vector<float> v;
        std::vector<int32_t> t;
        const int G = 60;
        for (int i = 0; i <= G; ++i)
            for (int j = 0; j <= G; ++j)
                for (float x : {-1 + 2.0f * i / G, 0.0f, -1 + 2.0f * j / G}) v.push_back(x);
        for (int i = 0; i < G; ++i)
            for (int j = 0; j < G; ++j) {
                const int a = i * (G + 1) + j;
                t.insert(t.end(), {a, a + 1, a + G + 2, a, a + G + 2, a + G + 1});
            }
        bad += check(v, t, 8000, 0.25f);
    }
    {  // 3,000 copies of one triangle: every hit is a tie
        std::vector<float> v;
        std::vector<int32_t> t;
        for (int i = 0; i < 9000; ++i) {
            t.push_back(i);
            for (int a = 0; a < 3; ++a) v.push_back(a == i % 3 ? 0.5f : 0.0f);
        }
        bad += check(v, t, 500, 0.0f);
    }
    if (!bad) std::puts("ok");
    return bad != 0;
}
