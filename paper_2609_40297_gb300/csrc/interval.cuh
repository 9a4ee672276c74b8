// The paper's screen-space overlap test of one sample against one ancestor (Sec. IV-B, Eq. 5-7),
// shared by the ray-by-ray count (interval.cu) and the per-node count (nodecount.cu). Every
// floating-point step is one correctly rounded single-precision operation (__fadd_rn and friends: no
// contraction), in a fixed order; the steps are described in interval.cu.
#pragma once

#include "dev_path.cuh"

namespace mig {
namespace dev {

constexpr float kZNear = 1.0f / 1024.0f;  // near end of the valid depth range, voxel units

struct Seg {
    float lo, hi;          // depth-clipped range of the ray fraction
    float Za, Zb;          // camera z at lo, hi (voxel units)
    float ua, va, ub, vb;  // projected clipped endpoints (pixels)
    float wa, wb;          // inverse depths at the endpoints
    float s0, s1;          // Liang-Barsky range of the screen parameter
    float ru, rv;          // reciprocals of the segment's screen extent (0 when it is 0)
};

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }

// The camera coordinates (Q32 to voxel units) of a point at offset r (Q16, exact integers) from an
// ancestor's camera with projection rows m (Q16: mu, mv, mz).
__device__ __forceinline__ float seg_coord(const int32_t *m, int rx, int ry, int rz) {
    const float sc = 2.3283064365386963e-10f;  // 2^-32: Q32 -> voxel units
    return fmul(__ll2float_rn((int64_t)m[0] * rx + (int64_t)m[1] * ry + (int64_t)m[2] * rz), sc);
}

// steps 1-3 for the candidate ray whose origin has camera coordinates (U0, V0, Z0) and whose range
// endpoint lies at r1 (Q16) from the ancestor with projection rows m; false if nothing of the ray is in
// view, or if the sample's ray fraction lam lies outside the depth-clipped range (seg_param would then
// reject it, so the screen-space part is skipped with the same outcome)
__device__ __forceinline__ bool seg_setup(const int32_t *m, float U0, float V0, float Z0, const int3 r1, float zf, int W, int H, float lam,
                                          Seg &g) {
    const float Z1 = seg_coord(m + 6, r1.x, r1.y, r1.z);
    const float zn = kZNear;
    const float dZ = fsub(Z1, Z0);
    float lo = 0.0f, hi = 1.0f;
    if (Z0 < zn) {
        if (!(dZ > 0.0f)) return false;
        lo = fdiv(fsub(zn, Z0), dZ);
    }
    if (Z1 < zn) {
        if (!(dZ < 0.0f)) return false;
        hi = fdiv(fsub(zn, Z0), dZ);
    }
    if (Z0 > zf) {
        if (!(dZ < 0.0f)) return false;
        const float l = fdiv(fsub(zf, Z0), dZ);
        if (l > lo) lo = l;
    }
    if (Z1 > zf) {
        if (!(dZ > 0.0f)) return false;
        const float h = fdiv(fsub(zf, Z0), dZ);
        if (h < hi) hi = h;
    }
    if (!(lo < hi)) return false;
    if (!(lam >= lo && lam <= hi)) return false;
    const float U1 = seg_coord(m, r1.x, r1.y, r1.z), V1 = seg_coord(m + 3, r1.x, r1.y, r1.z);
    const float dU = fsub(U1, U0), dV = fsub(V1, V0);
    const float Ua = fadd(U0, fmul(lo, dU)), Va = fadd(V0, fmul(lo, dV)), Za = fadd(Z0, fmul(lo, dZ));
    const float Ub = fadd(U0, fmul(hi, dU)), Vb = fadd(V0, fmul(hi, dV)), Zb = fadd(Z0, fmul(hi, dZ));
    if (!(Za > 0.0f && Zb > 0.0f)) return false;
    g.lo = lo;
    g.hi = hi;
    g.Za = Za;
    g.Zb = Zb;
    // Eq. 5 with the inverse depths of Eq. 6: u = U w, v = V w
    g.wa = fdiv(1.0f, Za);
    g.wb = fdiv(1.0f, Zb);
    g.ua = fmul(Ua, g.wa);
    g.va = fmul(Va, g.wa);
    g.ub = fmul(Ub, g.wb);
    g.vb = fmul(Vb, g.wb);
    // Liang-Barsky against 0 <= u <= W, 0 <= v <= H (edges in the order -u, +u, -v, +v); each
    // edge's crossing is q times the reciprocal of p
    const float du = fsub(g.ub, g.ua), dv = fsub(g.vb, g.va);
    g.ru = du != 0.0f ? fdiv(1.0f, du) : 0.0f;
    g.rv = dv != 0.0f ? fdiv(1.0f, dv) : 0.0f;
    const float pe[4] = {-du, du, -dv, dv};
    const float rp[4] = {-g.ru, g.ru, -g.rv, g.rv};
    const float qe[4] = {g.ua, fsub(__int2float_rn(W), g.ua), g.va, fsub(__int2float_rn(H), g.va)};
    float s0 = 0.0f, s1 = 1.0f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (pe[e] == 0.0f) {
            if (qe[e] < 0.0f) return false;
            continue;
        }
        const float r = fmul(qe[e], rp[e]);
        if (pe[e] < 0.0f) {
            if (r > s1) return false;
            if (r > s0) s0 = r;
        } else {
            if (r < s0) return false;
            if (r < s1) s1 = r;
        }
    }
    if (!(s0 < s1)) return false;
    g.s0 = s0;
    g.s1 = s1;
    return true;
}

// screen parameter of the ray fraction lam (perspective-correct); false outside the clip
__device__ __forceinline__ bool seg_param(const Seg &g, float lam, float &s) {
    if (!(lam >= g.lo && lam <= g.hi)) return false;
    const float mu = fdiv(fsub(lam, g.lo), fsub(g.hi, g.lo));
    const float num = fmul(mu, g.Zb);
    const float den = fadd(fmul(fsub(1.0f, mu), g.Za), num);
    s = fdiv(num, den);
    return s >= g.s0 && s < g.s1;
}

// a voxel's sample: midpoint of the ray's traversal of it (entry ne / ade, exit nx / adx capped at
// the range) as a fraction of the range T (= Tq / 2^30 in crossing units)
__device__ __forceinline__ float sample_lambda(uint32_t ne, uint32_t ade, uint32_t nx, uint32_t adx, float T) {
    const float lin = fdiv(fdiv(__uint2float_rn(ne), __uint2float_rn(ade)), T);
    float lout = fdiv(fdiv(__uint2float_rn(nx), __uint2float_rn(adx)), T);
    if (lout > 1.0f) lout = 1.0f;
    return fmul(fadd(lin, lout), 0.5f);
}

// Column (or row) crossings of the walk: boundary b_k = b0 + sgn k is crossed at screen parameter
// x(k) = (b_k - a0) * r, the walk's own formula, non-decreasing in k. Counts the crossings at or
// before s among k < kmax (crossing kmax leaves the buffer); lo / hi = the last crossing at or
// before s and the next one. The count starts from a float estimate and is corrected exactly.
__device__ __forceinline__ int count_crossings(float a0, float r, float d, int b0, int sgn, int kmax, float s,
                                               float &lo, float &hi) {
    const float est = (float)sgn * (s * d + a0 - (float)b0) + 1.0f;  // estimate only; corrected below
    int k = !(est > 0.0f) ? 0 : (est >= (float)kmax ? kmax : (int)est);
    auto x = [&](int kk) { return fmul(fsub(__int2float_rn(b0 + sgn * kk), a0), r); };
    while (k > 0 && x(k - 1) > s) --k;
    while (k < kmax && x(k) <= s) ++k;
    lo = k > 0 ? x(k - 1) : __int_as_float(0xff800000);
    hi = k < kmax ? x(k) : __int_as_float(0x7f800000);
    return k;
}

// Step 4 for one screen parameter s in [s0, s1): the walk's portion containing s, found directly.
// The walk crosses column and row boundaries in the order of their crossing parameters, so at s
// it is in column i0 + si * (column crossings <= s) and row j0 + sj * (row crossings <= s), in the
// portion from the latest crossing at or before s (s0 if none) to the next one (capped at s1).
// True if that portion is observed; false if not, or if the walk leaves the buffer before s.
__device__ __forceinline__ bool seg_lookup(const Seg &g, int W, int H, const uint32_t *D, float s MIG_CHECKED(, const LevelParams *p)) {
    const float du = fsub(g.ub, g.ua), dv = fsub(g.vb, g.va);
    const float ru = g.ru, rv = g.rv;
    const float fi = floorf(fadd(g.ua, fmul(g.s0, du))), fj = floorf(fadd(g.va, fmul(g.s0, dv)));
    const int i0 = fi < 0.0f ? 0 : (fi > __int2float_rn(W - 1) ? W - 1 : __float2int_rz(fi));
    const int j0 = fj < 0.0f ? 0 : (fj > __int2float_rn(H - 1) ? H - 1 : __float2int_rz(fj));
    const int si = du > 0.0f ? 1 : (du < 0.0f ? -1 : 0), sj = dv > 0.0f ? 1 : (dv < 0.0f ? -1 : 0);
    float xlo = __int_as_float(0xff800000), xhi = __int_as_float(0x7f800000), ylo = xlo, yhi = xhi;
    int nx = 0, ny = 0;
    if (si) {
        const int kmax = si > 0 ? W - i0 : i0 + 1;
        nx = count_crossings(g.ua, ru, du, si > 0 ? i0 + 1 : i0, si, kmax, s, xlo, xhi);
        if (nx == kmax) return false;
    }
    if (sj) {
        const int kmax = sj > 0 ? H - j0 : j0 + 1;
        ny = count_crossings(g.va, rv, dv, sj > 0 ? j0 + 1 : j0, sj, kmax, s, ylo, yhi);
        if (ny == kmax) return false;
    }
    const int i = i0 + si * nx, j = j0 + sj * ny;
    const float s_in = (nx == 0 && ny == 0) ? g.s0 : (xlo > ylo ? xlo : ylo);
    float s_out = xhi < yhi ? xhi : yhi;
    if (g.s1 < s_out) s_out = g.s1;
    const float sm = fmul(fadd(s_in, s_out), 0.5f);
    const float wm = fadd(g.wa, fmul(sm, fsub(g.wb, g.wa)));
#if MIG_DEBUG_BOUNDS
    const uint32_t *at = D + (size_t)j * W + i;
    if (p->arena_slots && !at_ok(*p, at, (const uint32_t *)p->arena, (size_t)p->arena_slots * W * H, kBoundsDepth)) return false;
#endif
    const float Dv = fmul(__uint2float_rn(ld_written(D + (size_t)j * W + i)), 1.52587890625e-05f);
    return fmul(wm, Dv) >= 1.0f;  // z <= D in inverse depth
}

}  // namespace dev
}  // namespace mig
