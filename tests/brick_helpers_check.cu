// Host checks of the brick steps (csrc/bricks.cuh, compiled for the host) against plain references
// written here:
//   cast  - cast_bricks (jumps through free space, exact voxel walk near occupied bricks) against a
//           plain DDA: step index and entry crossing of the first occupied voxel;
//   beam  - beam_free: the rays of a tile cast from where its beam stopped, against the same DDA;
//   box   - box_view: its verdict, depth bounds and pixel bounds against every voxel centre of the
//           box projected in exact integers (Eq. 5);
//   sure  - the certain visit (depth below zl2 / the yaw's zinf, distance below the range): the exact
//           visit test of the owner pixel's ray must agree for every voxel that is claimed;
//   slab  - visit_slab against the exact visit test.
// Usage: brick_helpers_check <seed>; prints one line of counts, exits 1 on any mismatch.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "bricks.cuh"

using namespace mig::dev;
typedef long long i64;

static i64 fdiv(i64 a, i64 b) {
    i64 q = a / b;
    return q - ((a % b != 0) && ((a < 0) != (b < 0)));
}

struct Grid {
    int N[3];
    std::vector<uint8_t> g;
    std::vector<uint64_t> om;
    std::vector<uint8_t> dist, oct[8];
    uint8_t at(int x, int y, int z) const { return g[((size_t)z * N[1] + y) * N[0] + x]; }
    void bricks() {
        const int b[3] = {(N[0] + 3) / 4, (N[1] + 3) / 4, (N[2] + 3) / 4};
        om.assign((size_t)b[0] * b[1] * b[2], 0);
        dist.assign(om.size(), kDistCap);
        for (int z = 0; z < N[2]; ++z)
            for (int y = 0; y < N[1]; ++y)
                for (int x = 0; x < N[0]; ++x)
                    if (at(x, y, z) == 2)
                        om[((size_t)(z / 4) * b[1] + y / 4) * b[0] + x / 4] |= 1ull << ((z % 4) * 16 + (y % 4) * 4 + x % 4);
        for (int o = 0; o < 8; ++o) {  // by definition: occupied bricks not behind along any axis
            const int s[3] = {o & 1 ? 1 : -1, o & 2 ? 1 : -1, o & 4 ? 1 : -1};
            oct[o].assign(om.size(), kDistCap);
            for (int z = 0; z < b[2]; ++z)
                for (int y = 0; y < b[1]; ++y)
                    for (int x = 0; x < b[0]; ++x) {
                        uint8_t &d = oct[o][((size_t)z * b[1] + y) * b[0] + x];
                        for (int k = 0; k < d; ++k)
                            for (int j = 0; j < d; ++j)
                                for (int i = 0; i < d; ++i) {
                                    const int X = x + s[0] * i, Y = y + s[1] * j, Z = z + s[2] * k;
                                    if (X < 0 || Y < 0 || Z < 0 || X >= b[0] || Y >= b[1] || Z >= b[2]) continue;
                                    if (om[((size_t)Z * b[1] + Y) * b[0] + X]) d = (uint8_t)std::min<int>(d, std::max(i, std::max(j, k)));
                                }
                        uint8_t &m = dist[((size_t)z * b[1] + y) * b[0] + x];
                        m = std::min(m, d);
                    }
        }
    }
};

// The DDA of Sec. IV-B: step index of the first occupied voxel (-1: none) and its entry crossing.
static int walk(const Grid &G, const i64 P[3], const i64 d[3], i64 Tq, i64 &en, i64 &ea) {
    i64 n[3], a[3];
    int v[3], s[3];
    for (int i = 0; i < 3; ++i) {
        v[i] = (int)fdiv(P[i], 65536);
        s[i] = d[i] < 0 ? -1 : 1;
        a[i] = std::llabs(d[i]);
        n[i] = d[i] < 0 ? P[i] - (i64)v[i] * 65536 : ((i64)v[i] + 1) * 65536 - P[i];
    }
    en = 0;
    ea = 1;
    for (int m = 0;; ++m) {
        if (G.at(v[0], v[1], v[2]) == 2) return m;
        int b = -1;
        for (int i = 0; i < 3; ++i)
            if (a[i] && (b < 0 || n[i] * a[b] < n[b] * a[i])) b = i;
        if (n[b] * (i64(1) << 30) >= Tq * a[b]) return -1;
        en = n[b];
        ea = a[b];
        v[b] += s[b];
        if (v[b] < 0 || v[b] >= G.N[b]) return -1;
        n[b] += 65536;
    }
}

int main(int argc, char **argv) {
    std::mt19937_64 rng(argc > 1 ? atoi(argv[1]) : 1);
    auto uni = [&](double lo, double hi) { return lo + (hi - lo) * ((rng() >> 11) * (1.0 / 9007199254740992.0)); };
    i64 rays = 0, hits = 0, cast_bad = 0, boxes = 0, in1 = 0, out1 = 0, box_bad = 0;
    i64 beam_rays = 0, beam_free_rays = 0, beam_bad = 0;
    i64 sure = 0, cand = 0, sure_bad = 0, slabs = 0, undecided = 0, slab_bad = 0;

    // ---- cast
    for (int trial = 0; trial < 60; ++trial) {
        Grid G;
        for (int i = 0; i < 3; ++i) G.N[i] = trial % 9 == 0 ? 1 + (int)(rng() % 9) : 1 + (int)(rng() % (i == 2 ? 60 : 170));
        if (trial % 7 == 3) G.N[0] = 900 + (int)(rng() % 300), G.N[1] = 5 + (int)(rng() % 9), G.N[2] = 5 + (int)(rng() % 9);
        G.g.assign((size_t)G.N[0] * G.N[1] * G.N[2], 1);
        const double po[5] = {0.0, 0.00003, 0.0005, 0.005, 0.05};
        for (auto &c : G.g) c = uni(0, 1) < po[trial % 5] ? 2 : (uint8_t)(rng() & 1);
        G.bricks();
        for (int r = 0; r < 2500; ++r) {
            i64 P[3], d[3];
            double q[3], nr = 0;
            for (int i = 0; i < 3; ++i) {
                const int m = (int)(rng() % 6);
                const i64 v = (i64)(rng() % G.N[i]);
                P[i] = m == 0 ? v * 65536 : m == 1 ? v * 65536 + 32768 : m == 2 ? (v / 4 * 4) * 65536 : m == 3 ? v * 65536 + 65535 : v * 65536 + (i64)(rng() % 65536);
                q[i] = uni(-1, 1);
            }
            const int m = (int)(rng() % 8);
            if (m == 0) q[rng() % 3] = 0;
            if (m == 1) q[0] = q[1] = 0.5, q[2] = rng() % 2 ? 0.5 : 0;
            if (m == 2) q[0] = rng() & 1 ? 1 : -1, q[1] = q[2] = 0;
            if (m == 3) q[rng() % 3] *= 1e-5;
            if (m == 4) q[rng() % 3] *= 1e-8, q[rng() % 3] *= 1e-3;
            for (int i = 0; i < 3; ++i) nr += q[i] * q[i];
            if (nr < 1e-12) continue;
            for (int i = 0; i < 3; ++i) d[i] = llrint(q[i] / std::sqrt(nr) * 1073741824.0);
            if (rng() % 4 == 0)
                for (int i = 0; i < 3; ++i) d[i] = d[i] / 1024 * 1024;
            if (!d[0] && !d[1] && !d[2]) continue;
            const i64 Tq = (i64)(rng() % ((trial % 7 == 3 ? 1024 : 200) * 65536)) + 1;
            i64 en, ea;
            const int w = walk(G, P, d, Tq, en, ea);
            uint32_t ne, ade, f = 0, c = 0;
            const uint32_t got = cast_bricks<true, false>(G.om.data(), G.oct[octant_of((int)d[0], (int)d[1], (int)d[2])].data(), G.N[0], G.N[1], G.N[2], (int)P[0], (int)P[1],
                                                          (int)P[2], (int)d[0], (int)d[1], (int)d[2], Tq, 0.0f, ne, ade, f, c);
            ++rays;
            hits += w >= 0;
            if (got != (w < 0 ? kNoHit : (uint32_t)w) || (w >= 0 && ((i64)ne != en || (i64)ade != ea))) ++cast_bad;
        }
    }

    // ---- beams: an 8x4 tile of a pinhole camera; every ray starts where the tile's beam stopped
    for (int trial = 0; trial < 90; ++trial) {
        Grid G;
        for (int i = 0; i < 3; ++i) G.N[i] = 1 + (int)(rng() % (i == 2 ? 60 : 170));
        G.g.assign((size_t)G.N[0] * G.N[1] * G.N[2], 1);
        const double po[4] = {0.00001, 0.0001, 0.001, 0.01};
        for (auto &c : G.g) c = uni(0, 1) < po[trial % 4] ? 2 : (uint8_t)(rng() & 1);
        G.bricks();
        const double th = uni(0.2, 2.5), tv = uni(0.2, 2.0), pitch = trial % 2 ? 0 : uni(-0.7, 0.7), cp = std::cos(pitch), sp = std::sin(pitch);
        const int W = 1 + (int)(rng() % 320), H = 1 + (int)(rng() % 240);
        for (int r = 0; r < 120; ++r) {
            i64 P[3];
            for (int i = 0; i < 3; ++i) P[i] = r % 5 ? (i64)(rng() % ((i64)G.N[i] * 65536)) : (i64)(rng() % G.N[i]) * 65536;
            const double yaw = r % 4 ? uni(0, 6.3) : (r % 16) / 4 * M_PI / 2, cs = std::cos(yaw), sn = std::sin(yaw);
            const i64 Tq = (i64)(rng() % (170 * 65536)) + 1;
            const int i0 = (int)(rng() % W) / 8 * 8, j0 = (int)(rng() % H) / 4 * 4, i1 = std::min(i0 + 7, W - 1), j1 = std::min(j0 + 3, H - 1);
            auto dir = [&](int i, int j, double w[3]) {  // over camera depth
                const double a = ((double)(2 * i + 1 - W) / W) * th, b = ((double)(2 * j + 1 - H) / H) * tv;
                const double f = cp - b * sp, l = -a;
                w[0] = cs * f - sn * l;
                w[1] = sn * f + cs * l;
                w[2] = -(b * cp + sp);
                return std::sqrt(a * a + b * b + 1.0);
            };
            float lo[3] = {1e30f, 1e30f, 1e30f}, hi[3] = {-1e30f, -1e30f, -1e30f};
            double cz = 0;
            for (int j = j0; j <= j1; ++j)
                for (int i = i0; i <= i1; ++i) {
                    double w[3];
                    const double nrm = dir(i, j, w);
                    cz = std::max(cz, 1.0 / nrm);
                    if ((i == i0 || i == i1) && (j == j0 || j == j1))
                        for (int a = 0; a < 3; ++a) lo[a] = std::min(lo[a], (float)w[a]), hi[a] = std::max(hi[a], (float)w[a]);
                }
            const float s = beam_free(G.dist.data(), G.N[0], G.N[1], G.N[2], (int)P[0], (int)P[1], (int)P[2], lo, hi,
                                      (float)(Tq / 65536.0 * cz * 1.00001));
            for (int j = j0; j <= j1; ++j)
                for (int i = i0; i <= i1; ++i) {
                    double w[3];
                    const double nrm = dir(i, j, w);
                    i64 d[3], en, ea;
                    for (int a = 0; a < 3; ++a) d[a] = llrint(w[a] / nrm * 1073741824.0);
                    const int want = walk(G, P, d, Tq, en, ea);
                    uint32_t got = kNoHit, ne, ade, f = 0, c = 0;
                    const float t0 = s > 0 ? std::max(0.0f, (float)(s * nrm) * (1.0f - 1e-6f) - kCastEps) : 0.0f;
                    if (s < 1e29f)
                        got = cast_bricks<true, false>(G.om.data(), G.oct[octant_of((int)d[0], (int)d[1], (int)d[2])].data(), G.N[0], G.N[1], G.N[2], (int)P[0], (int)P[1], (int)P[2],
                                                       (int)d[0], (int)d[1], (int)d[2], Tq, t0, ne, ade, f, c);
                    ++beam_rays;
                    beam_free_rays += s >= 1e29f;
                    if (got != (want < 0 ? kNoHit : (uint32_t)want) || (want >= 0 && s < 1e29f && ((i64)ne != en || (i64)ade != ea))) ++beam_bad;
                }
        }
    }

    // ---- boxes and visits
    for (int trial = 0; trial < 500; ++trial) {
        const int W = trial % 9 == 0 ? 1 + (int)(rng() % 4) : trial % 11 == 0 ? 2048 : 1 + (int)(rng() % 400);
        const int H = trial % 7 == 0 ? 1 + (int)(rng() % 4) : 1 + (int)(rng() % 300);
        const double hf = trial % 5 == 0 ? uni(5, 175) : uni(40, 110), vf = trial % 5 == 1 ? uni(5, 175) : uni(30, 80);
        const double pitch = trial % 3 ? (trial % 3 == 1 ? 0.0 : uni(-25, 25)) : uni(-90, 90);
        const int K = 1 + (int)(rng() % 48), k = trial % 4 ? (int)(rng() % K) : 0;
        const double th = std::tan(hf * 0.5 * M_PI / 180), tv = std::tan(vf * 0.5 * M_PI / 180);
        const double cp = std::cos(pitch * M_PI / 180), sp = std::sin(pitch * M_PI / 180);
        const double fx = W * 0.5 / th, fy = H * 0.5 / tv, cs = std::cos(2 * M_PI * k / K), sn = std::sin(2 * M_PI * k / K);
        const double ex[3] = {sn, -cs, 0}, ey[3] = {-sp * cs, -sp * sn, -cp}, ez[3] = {cp * cs, cp * sn, -sp};
        int32_t row[12] = {(int32_t)llrint(cs * 1073741824.0), (int32_t)llrint(sn * 1073741824.0)};
        bool ok = true;
        for (int a = 0; a < 3; ++a) {
            const double mu = fx * ex[a] + W * 0.5 * ez[a], mv = fy * ey[a] + H * 0.5 * ez[a];
            ok = ok && std::fabs(mu) * 65536 < 2147483647.0 && std::fabs(mv) * 65536 < 2147483647.0;
            if (!ok) break;
            row[2 + a] = (int32_t)llrint(mu * 65536);
            row[5 + a] = (int32_t)llrint(mv * 65536);
            row[8 + a] = (int32_t)llrint(ez[a] * 65536);
        }
        if (!ok) continue;
        const VisitLimits vl = visit_limits(hf, vf, W, H);
        const YawRows yr = yaw_rows(row, W, H, vl.hu, vl.hv, (float)(1 / fx), (float)(1 / fy));
        const int R = trial % 2 ? 10 + (int)(rng() % 160) : 10 + (int)(rng() % 1010);
        const i64 Tq = (i64)R * 65536 - (i64)(rng() % 65536);
        const float Tvox = (float)Tq / 65536.0f;
        const int big[3] = {8, 8, 4}, small[3] = {2, 2, 2};
        for (int bi = 0; bi < 400; ++bi) {
            i64 P[3];
            for (int a = 0; a < 3; ++a) P[a] = (i64)(rng() % (2000ll * 65536)) + 1050ll * 65536;
            // a box somewhere about the view (or anywhere) within the range
            const double u = uni(-1.3, 1.3) * th, v = uni(-1.3, 1.3) * tv, z = uni(0, 1) * R / std::sqrt(1 + u * u + v * v);
            const bool any = rng() % 6 == 0;
            const int *half = bi % 3 ? small : big;
            int o[3];  // first voxel of the box
            for (int a = 0; a < 3; ++a) {
                const double c = any ? uni(-R, R) : z * (u * ex[a] + v * ey[a] + ez[a]);
                o[a] = (int)std::floor(P[a] / 65536.0 + c) / 4 * 4 - half[a] + 2;
            }
            float c[3];
            for (int a = 0; a < 3; ++a) c[a] = (float)(int)(((i64)(o[a] + half[a]) << 16) - P[a]) / 65536.0f;
            const float h[3] = {half[0] - 0.5f, half[1] - 0.5f, half[2] - 0.5f};
            const BoxView b = bi % 3 ? box_view<true>(yr, c[0], c[1], c[2], h[0], h[1], h[2], W, H) : box_view<false>(yr, c[0], c[1], c[2], h[0], h[1], h[2], W, H);
            ++boxes;
            in1 += b.in > 0;
            out1 += b.in < 0;
            float far = 0;
            for (int a = 0; a < 3; ++a) far += (std::fabs(c[a]) + h[a]) * (std::fabs(c[a]) + h[a]);
            far = std::sqrt(far);
            const bool sv = b.in >= 0 && b.zlo >= 0.5f &&
                            ((b.zhi < yr.x.x && far + 0.86f < Tvox) || (b.zhi < vl.zl2 && far + 0.02f < Tvox));
            for (int dz = 0; dz < 2 * half[2]; ++dz)
                for (int dy = 0; dy < 2 * half[1]; ++dy)
                    for (int dx = 0; dx < 2 * half[0]; ++dx) {
                        const int vx[3] = {o[0] + dx, o[1] + dy, o[2] + dz};
                        i64 r[3];
                        for (int a = 0; a < 3; ++a) r[a] = ((i64)vx[a] << 16) + 32768 - P[a];
                        const i64 Z = row[8] * r[0] + row[9] * r[1] + row[10] * r[2];
                        const i64 U = row[2] * r[0] + row[3] * r[1] + row[4] * r[2];
                        const i64 V = row[5] * r[0] + row[6] * r[1] + row[7] * r[2];
                        const double zv = (double)Z / 4294967296.0;
                        bool in = false;
                        i64 pu = -1, pv = -1;
                        if (Z > 0) {
                            pu = fdiv(U, Z);
                            pv = fdiv(V, Z);
                            in = pu >= 0 && pu < W && pv >= 0 && pv < H;
                        }
                        if ((b.in < 0 && in) || (b.in > 0 && !in)) ++box_bad;
                        if (b.in >= 0 && (zv < b.zlo || zv > b.zhi)) ++box_bad;
                        if (b.in >= 0 && b.zlo >= 0.5f && in && (pu < b.u0 || pu > b.u1 || pv < b.v0 || pv > b.v1)) ++box_bad;
                        if (!in || (bi % 3 == 0 && (rng() & 7))) continue;
                        // the owner ray: the body-frame ray of the pixel, rotated by the yaw
                        const double a_ = ((double)(2 * pu + 1 - W) / W) * th, b_ = ((double)(2 * pv + 1 - H) / H) * tv;
                        const double nrm = std::sqrt(a_ * a_ + b_ * b_ + 1.0);
                        const int4 body = make_int4((int)llrint((cp - b_ * sp) / nrm * 1073741824.0), (int)llrint(-a_ / nrm * 1073741824.0),
                                                    (int)llrint(-(b_ * cp + sp) / nrm * 1073741824.0), (int)llrint(1073741824.0 / nrm));
                        const int ddx = (int)(((i64)row[0] * body.x - (i64)row[1] * body.y) >> 30),
                                  ddy = (int)(((i64)row[1] * body.x + (i64)row[0] * body.y) >> 30);
                        const bool vis = visit_index((int)P[0], (int)P[1], (int)P[2], ddx, ddy, body.z, vx[0], vx[1], vx[2], Tq) >= 0;
                        ++cand;
                        sure += sv;
                        if (sv && !vis) ++sure_bad;
                        const float q = 1.0f / 1073741824.0f, ck = (float)row[0] * q, sk = (float)row[1] * q;
                        const float bxf = (float)body.x * q, byf = (float)body.y * q;
                        const int s = visit_slab((float)(int)r[0] / 65536.0f, (float)(int)r[1] / 65536.0f, (float)(int)r[2] / 65536.0f,
                                                 ck * bxf - sk * byf, sk * bxf + ck * byf, (float)body.z * q, Tvox);
                        ++slabs;
                        undecided += s < 0;
                        if (s >= 0 && (s > 0) != vis) ++slab_bad;
                    }
        }
    }
    printf("rays %lld hits %lld cast_bad %lld beam_rays %lld beam_free %lld beam_bad %lld boxes %lld inside %lld outside %lld box_bad %lld visits %lld sure %lld sure_bad %lld "
           "slabs %lld undecided %lld slab_bad %lld\n",
           rays, hits, cast_bad, beam_rays, beam_free_rays, beam_bad, boxes, in1, out1, box_bad, cand, sure, sure_bad, slabs, undecided, slab_bad);
    return (cast_bad || beam_bad || box_bad || sure_bad || slab_bad) ? 1 : 0;
}
