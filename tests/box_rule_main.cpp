// The four-wide walk on the CPU with the library's own box and stack rules (gsp_reach, gsp_wide_keep,
// gsp_wide_entry), a lane's steps as csrc/wide.cuh makes them, against every triangle in turn: the same
// triangle and t, whatever tmin, the length of the direction, and the last bit of the reciprocals (which
// the device takes from an approximation). Lines (tmin far behind the origin) cost what long rays cost.
// Arguments: the group of cases (tests/test_box_rule.py); "links" for the library's walk of the hit/miss links.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "gsp_internal.h"

static int32_t as_int(float f) { int32_t i; std::memcpy(&i, &f, 4); return i; }
static float as_float(int32_t i) { float f; std::memcpy(&f, &i, 4); return f; }

static const int32_t kNone = INT32_MIN, kMiss = 0x7fffffff;

struct Mesh {
    std::vector<float> v;
    std::vector<int32_t> t;
};

struct Best {
    float t;
    int32_t id;
};

// Moller-Trumbore on one triangle {v0, id}, {v1, .}, {v2, .}
static void test_tri(const float4* tri, const float* r, Best& b) {
    const float *P = (const float*)tri, *d = r + 4;
    float e1[3], e2[3], s[3];
    for (int a = 0; a < 3; ++a) {
        e1[a] = P[4 + a] - P[a];
        e2[a] = P[8 + a] - P[a];
        s[a] = r[a] - P[a];
    }
    const float px = d[1] * e2[2] - d[2] * e2[1], py = d[2] * e2[0] - d[0] * e2[2], pz = d[0] * e2[1] - d[1] * e2[0];
    const float det = e1[0] * px + e1[1] * py + e1[2] * pz;
    if (det == 0) return;
    const float f = 1.0f / det, u = f * (s[0] * px + s[1] * py + s[2] * pz);
    const float qx = s[1] * e1[2] - s[2] * e1[1], qy = s[2] * e1[0] - s[0] * e1[2], qz = s[0] * e1[1] - s[1] * e1[0];
    const float v = f * (d[0] * qx + d[1] * qy + d[2] * qz), t = f * (e2[0] * qx + e2[1] * qy + e2[2] * qz);
    const int32_t id = as_int(P[3]);
    if (u >= 0 && v >= 0 && u + v <= 1 && t > r[3] && (t < b.t || (t == b.t && b.id >= 0 && id < b.id))) b = {t, id};
}

template <bool BEHIND>
static Best walk(const HostBVH& b, const std::vector<float4>& wide, const float* r, int ulp, int64_t& nodes) {
    const float *W = (const float*)wide.data(), *d = r + 4;
    float inv[3];
    for (int k = 0; k < 3; ++k) inv[k] = as_float(as_int(1.0f / (std::fabs(d[k]) < 1e-30f ? std::copysign(1e-30f, d[k]) : d[k])) + ulp);
    Best best{r[7], -1};
    struct { int32_t key, ref; } stk[64];
    int32_t cur = 0;
    int sp = 0;
    const auto pop = [&] {
        while (sp > 0) {
            --sp;
            if (gsp_wide_keep<BEHIND>(stk[sp].key, best.t)) return stk[sp].ref;
        }
        return kNone;
    };
    while (cur != kNone) {
        if (cur < 0) {
            for (int k = 0; k < (~cur & 7); ++k) test_tri(&b.tris[3 * ((~cur >> 3) + k)], r, best);
            cur = pop();
            continue;
        }
        ++nodes;
        const float* q = W + 32 * (int64_t)cur;
        int32_t key[4], nearest = kMiss;
        for (int c = 0; c < 4; ++c) {
            float tn = r[3], tf = INFINITY;
            for (int k = 0; k < 3; ++k) {
                const float tc = (q[8 * k + c] - r[k]) * inv[k], h = q[8 * k + 4 + c], a = std::fabs(inv[k]);
                tn = std::fmax(tn, std::fmaf(-h, a, tc));
                tf = std::fmin(tf, std::fmaf(h, a, tc));
            }
            key[c] = tn <= gsp_reach<BEHIND>(std::fmin(best.t, tf)) ? ((gsp_wide_order<BEHIND>(tn) & ~3) | c) : kMiss;
            nearest = std::min(nearest, key[c]);
        }
        if (nearest == kMiss) {
            cur = pop();
            continue;
        }
        for (int c = 0; c < 4; ++c)
            if (key[c] != kMiss && key[c] != nearest) {
                if (sp == 64) return {0.0f, -2};
                stk[sp].key = key[c];
                stk[sp++].ref = as_int(q[24 + c]);
            }
        cur = as_int(q[24 + (nearest & 3)]);
    }
    return best;
}

static bool links;  // the library's host walk of the hit/miss links instead

// nr rays from the box around `at` with half extent 2 `size`, directions of length about `len`. Returns
// the number of rays whose walk differs from the triangles in turn.
static int check(const char* name, const Mesh& m, int nr, float at, float size, float len) {
    const int nt = (int)m.t.size() / 3;
    HostBVH b;
    if (!bvh_build_host(m.v.data(), (int64_t)m.v.size() / 3, m.t.data(), nt, gsp_bvh_params{16, 4, 7, 6}, b).empty()) return 1;
    std::vector<float4> wide((size_t)b.nwide * 8);
    for (int64_t i = 0; i < (int64_t)b.wide_of.size(); ++i)
        if (b.wide_of[i] >= 0) gsp_wide_entry(b.bin.data(), i, [&](int32_t j) { return b.wide_of[j]; }, &wide[8 * b.wide_of[i]]);
    int bad = 0;
    // -16 size / len: behind everything that a ray's line meets
    const float behind = -16.0f * size / len;
    int64_t cost[6] = {}, line = 0, moved = 0;
    const float tmins[6] = {0.0f, behind / 16, behind, 1e6f * behind, -FLT_MAX, -INFINITY};
    for (int j = 0; j < 6; ++j) {
        std::mt19937 g(nt);
        std::uniform_real_distribution<float> u(-1.0f, 1.0f);
        int wrong = 0, hits = 0;
        for (int i = 0; i < nr; ++i) {
            float r[8], n = 0;
            for (int k = 0; k < 3; ++k) {
                r[k] = at + 2 * size * u(g);
                do r[4 + k] = u(g);
                while (std::fabs(r[4 + k]) < 0.2f);  // no component of a short direction falls below 1e-30
                n += r[4 + k] * r[4 + k];
            }
            for (int k = 0; k < 3; ++k) r[4 + k] = r[4 + k] / std::sqrt(n) * len;
            r[3] = tmins[j];
            r[7] = i % 3 ? INFINITY : size / len;
            Best want{r[7], -1};
            for (int k = 0; k < nt; ++k) test_tri(&b.tris[3 * k], r, want);
            hits += want.id >= 0;
            if (links) {
                Best got;
                int32_t visits;
                bvh_host_walk(b, r, 1, &got.id, &got.t, &visits, nullptr);
                cost[j] += visits;
                wrong += got.id != want.id || (want.id >= 0 && got.t != want.t);
            }
            for (int ulp = -1; ulp <= 1 && !links; ++ulp) {
                const Best got = walk<true>(b, wide, r, ulp, cost[j]);
                wrong += got.id != want.id || (want.id >= 0 && got.t != want.t);
                if (tmins[j] < 0) continue;
                int64_t nodes = 0;  // the rays in front of the origin have a form of the rules of their own
                const Best ahead = walk<false>(b, wide, r, ulp, nodes);
                wrong += ahead.id != got.id || (got.id >= 0 && ahead.t != got.t);
            }
            if (j == 2 && !links) {  // the same line from where it starts
                walk<true>(b, wide, r, 0, line);
                for (int k = 0; k < 3; ++k) r[k] += behind * r[4 + k];
                r[3] = 0.0f;
                r[7] -= behind;
                walk<false>(b, wide, r, 0, moved);
            }
        }
        if (wrong || !hits) std::printf("%s, direction %g, tmin %g: %d of %d walks wrong, %d hits\n", name, len, tmins[j], wrong, links ? nr : 3 * nr, hits);
        bad += wrong + !hits;
    }
    if (line > 1.05 * moved) {  // the nearest box first and the far ones dropped, behind the origin too
        std::printf("%s, direction %g: %lld nodes from behind, %lld from a start there\n", name, len, (long long)line, (long long)moved);
        ++bad;
    }
    for (int j = 3; j < 6; ++j)  // the boxes a line meets do not depend on where far behind it starts
        if (cost[j] > 1.05 * cost[2]) {
            std::printf("%s, direction %g, tmin %g: %lld nodes, %lld at %g\n", name, len, tmins[j], (long long)cost[j], (long long)cost[2], behind);
            ++bad;
        }
    return bad;
}

static Mesh soup(int nt, float at, float size) {
    Mesh m;
    std::mt19937 g(nt);
    std::uniform_real_distribution<float> u(-1.0f, 1.0f);
    for (int i = 0; i < 3 * nt; ++i) m.t.push_back(i);
    for (int i = 0; i < nt; ++i) {
        const float c[3] = {u(g), u(g), u(g)};
        for (int k = 0; k < 9; ++k) m.v.push_back(at + size * (c[k % 3] + 0.2f * u(g)));
    }
    return m;
}

// A G x G grid of squares at height y: its boxes have no extent along one axis
static void add_floor(Mesh& m, int G, float y, float shift) {
    const int base = (int)m.v.size() / 3;
    for (int i = 0; i <= G; ++i)
        for (int j = 0; j <= G; ++j)
            for (float x : {-1 + 2.0f * i / G + shift, y, -1 + 2.0f * j / G + shift}) m.v.push_back(x);
    for (int i = 0; i < G; ++i)
        for (int j = 0; j < G; ++j) {
            const int a = base + i * (G + 1) + j;
            m.t.insert(m.t.end(), {a, a + 1, a + G + 2, a, a + G + 2, a + G + 1});
        }
}

int main(int argc, char** argv) {
    const std::string group = argc > 1 ? argv[1] : "";
    links = argc > 2 && std::string(argv[2]) == "links";
    int bad = 0;
    if (group == "tmin") {
        for (float len : {1.0f, 20.0f, 0.05f}) {
            for (int nt : {6, 40, 2000}) bad += check("soup", soup(nt, 0.0f, 1.0f), 1500, 0.0f, 1.0f, len);
            Mesh floor;
            add_floor(floor, 30, 0.0f, 0.0f);
            bad += check("floor", floor, 1500, 0.0f, 1.0f, len);
        }
        // distances that overflow for the box of an absent child, at the origin, but not for the scene's
        bad += check("far away, short directions", soup(300, -1e10f, 1e7f), 1500, -1e10f, 1e7f, 1e-29f);
    }
    if (group == "ties") {
        for (float len : {1.0f, 20.0f, 0.05f}) {
            Mesh floors;  // two floors at one height, differently divided
            add_floor(floors, 30, 0.3f, 0.0f);
            add_floor(floors, 23, 0.3f, 0.013f);
            bad += check("two floors", floors, 1500, 0.0f, 1.0f, len);
            for (float slope : {0.0f, 0.5f}) {  // triangles over one another in one plane
                Mesh m = soup(2000, 0.0f, 1.0f);
                for (size_t i = 0; i < m.v.size(); i += 3) m.v[i + 1] = 0.37f + slope * m.v[i] - 0.5f * slope * m.v[i + 2];
                bad += check("one plane", m, 1500, 0.0f, 1.0f, len);
            }
        }
    }
    if (!bad) std::puts("ok");
    return bad != 0;
}
