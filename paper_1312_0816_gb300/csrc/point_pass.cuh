// point_pass.cuh -- Contains and Safety of one point per lane over every
// daughter of a volume of boxes, tubes and cones, from the filter's tables
// (filter_pass.cuh: cheap tests of all daughters together, then each lane's
// own solids), and the FP64 work left: one feature of one solid.
//
// Contains.  A solid whose inflated copy does not hold the FP32 point does not
// hold the exact one; one whose copy shrunk by 2 delta holds it surely does.  Only
// between the two (a few in 10^5 points) FP64 decides.
//
// Safety.  Every solid gets an FP32 lower bound of its distance, the mother of
// its inside distance; the three least are kept.  The solid with the least
// bound is evaluated in FP64, and when the second bound exceeds that value by
// more than the FP64 rounding it is the minimum (queries.cuh).  The whole FP64
// routine tries every feature of a solid (a cone's four edges with a square
// root and a division each).  Here the FP32 point says in which zone of the
// solid it lies -- nearest to a plane, to a radius, to an edge or corner --
// with 2 delta to spare on every side, and FP64 forms that distance alone.  The
// routine's other terms are then 0 (a clamp) or larger by far more
// than their rounding (another edge), and where it takes the square root of a
// single square, the root is that number itself (sqrt(fl(x^2)) = |x| in
// binary64 rounded to nearest, without underflow), so the bits are the
// routine's.
#pragma once
#include "filter_pass.cuh"
#include "geo_internal.h"
#include "nav_common.cuh"
#include "queries.cuh"
#include "shapes32.cuh"
#include "shapes64.cuh"

namespace geonav {

// Zones of a point with respect to a solid: none (not certain), the plane of
// axis kZonePlane + k, the outer or inner radius, a corner (a box's edge or corner too),
// a cone's slanted edge, surely inside.
enum : int {
    kZoneNone = 0, kZonePlane = 1, kZoneOuter = 4, kZoneInner = 5, kZoneCorner = 6, kZoneSlant = 10, kZoneInside = 12
};
// kZoneCorner + (1 inner) + (2 at +dz); kZoneSlant + (1 inner)

// local coordinates of the FP32 point
__device__ __forceinline__ void point_to_entry(const float4* H, const float4 h0, int flags, float r8, const float* p,
                                               float* x) {
    const float w[3] = {p[0] - h0.x, p[1] - h0.y, p[2] - h0.z};
    if (flags & kFiltIdentity) {
        x[0] = w[0]; x[1] = w[1]; x[2] = w[2];
    } else {
        rotate_in(H[1], H[2], r8, w, x);
    }
}

// 0: surely outside solid h, 1: surely inside, 2: between
__device__ __forceinline__ int entry_holds(const FiltHvy* h, const float* p) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h3 = H[3], h4 = H[4];
    const int flags = __float_as_int(h3.y);
    float x[3];
    point_to_entry(H, h0, flags, h3.x, p, x);
    if (flags & kFiltBox) {
        const float a = fabsf(x[0]) - h4.x, b = fabsf(x[1]) - h4.y, c = fabsf(x[2]) - h4.z;
        const float m = fmaxf(a, fmaxf(b, c));
        return m > 0.f ? 0 : (m <= -2.f * h4.w ? 1 : 2);
    }
    const float4 h5 = H[5], h6 = H[6];
    const float rho2 = fmaf(x[0], x[0], x[1] * x[1]), az = fabsf(x[2]), g = h6.y;
    const bool hole = (flags & kFiltHole) != 0;
    const float ro = fmaf(h4.z, x[2], h4.y), ri = fmaf(h5.x, x[2], h4.w);
    if (az > h4.x || rho2 > ro * ro || (hole && rho2 < ri * ri)) return 0;
    const float si = ro - g, so = ri + g;
    return !(flags & kFiltLoose) && az <= h4.x - g && si > 0.f && rho2 <= si * si && (!hole || rho2 >= so * so) ? 1 : 2;
}

// Lower bound of the distance to solid h (0 inside its copy), lowered by the
// relative margin of the safety bounds.
__device__ __forceinline__ float entry_distance(const FiltHvy* h, const float* p) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h3 = H[3], h4 = H[4];
    const int flags = __float_as_int(h3.y);
    float x[3];
    point_to_entry(H, h0, flags, h3.x, p, x);
    float s;
    if (flags & kFiltBox) {
        const float a = fmaxf(fabsf(x[0]) - h4.x, 0.f), b = fmaxf(fabsf(x[1]) - h4.y, 0.f),
                    c = fmaxf(fabsf(x[2]) - h4.z, 0.f);
        s = fsqrt(fmaf(a, a, fmaf(b, b, c * c)));
    } else {
        const float bi = H[5].x;
        const float rho = fsqrt(fmaf(x[0], x[0], x[1] * x[1]));
        const float dz = fabsf(x[2]) - h4.x;
        const float so = rho - fmaf(h4.z, x[2], h4.y);
        const float si = (flags & kFiltHole) ? fmaf(bi, x[2], h4.w) - rho : -1.f;
        if (h4.z == 0.f && bi == 0.f) {
            const float dr = fmaxf(fmaxf(so, si), 0.f), d = fmaxf(dz, 0.f);
            s = fsqrt(fmaf(dr, dr, d * d));
        } else {
            s = fmaxf(fmaxf(dz, so * frsqrt(fmaf(h4.z, h4.z, 1.f))), fmaxf(si * frsqrt(fmaf(bi, bi, 1.f)), 0.f));
        }
    }
    return s * (1.f - kSafMargin);
}

// The zone of a point outside solid h (or surely inside it).  Every comparison
// keeps 2 delta (times the slope's factor) from the solid's own limit, which
// is the copy's less delta.  Of a point `grow` times beyond the extent that the copy
// was made for, the FP32 rounding is that much larger, and so is what they keep.
__device__ __forceinline__ int entry_zone(const FiltHvy* h, const float* p, const float grow = 1.f) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h3 = H[3], h4 = H[4];
    const int flags = __float_as_int(h3.y);
    float x[3];
    point_to_entry(H, h0, flags, h3.x, p, x);
    if (flags & kFiltBox) {
        const float d = h4.w * grow;
        const float e[3] = {fabsf(x[0]) - h4.x, fabsf(x[1]) - h4.y, fabsf(x[2]) - h4.z};   // less delta
        int out = 0, in = 0, k = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const bool o = e[q] > d, i = e[q] < -3.f * d;
            k = o ? q : k;
            out += o;
            in += i;
        }
        if (in == 3) return kZoneInside;
        if (out == 0) return kZoneNone;
        return out == 1 && in == 2 ? kZonePlane + k : kZoneCorner;
    }
    if (flags & kFiltLoose) return kZoneNone;
    const float4 h5 = H[5], h6 = H[6];
    const float m = h6.y * grow;   // 2 delta sqrt(1 + slope^2)
    const bool hole = (flags & kFiltHole) != 0;
    const float rho = fsqrt(fmaf(x[0], x[0], x[1] * x[1]));
    const float z = x[2], az = fabsf(z), dz = h4.x - h6.z;
    const float bo = h4.z, bi = h5.x, half = 0.5f * h6.y;
    const float ao = h4.y - half, ai = h4.w + half;   // the solid's own radius lines, to delta
    const float no = rho - fmaf(bo, z, ao), ni = hole ? fmaf(bi, z, ai) - rho : -1e30f;   // > 0: outside, in the hole
    const float zc = az - dz;
    if (zc < -m && no < -m && ni < -m) return kZoneInside;
    if (bo == 0.f && bi == 0.f) {   // a tube
        const bool beyond = zc > m, within = zc < -m;
        const bool o = no > m, i = ni > m, ring = no < -m && ni < -m;
        if (beyond) return ring ? kZonePlane + 2 : (o ? kZoneCorner : (i ? kZoneCorner + 1 : kZoneNone));
        if (within) return o ? kZoneOuter : (i ? kZoneInner : kZoneNone);
        return kZoneNone;
    }
    // a cone: its meridian section is a convex trapezoid, and the nearest
    // feature is the edge whose normal strip, or the vertex whose normal cone,
    // holds the point
    const float ze = copysignf(dz, z);
    if (zc > m && rho < fmaf(bo, ze, ao) - m && (!hole || rho > fmaf(bi, ze, ai) + m)) return kZonePlane + 2;
    const float po = fmaf(bo, rho - ao, z) * frcp(fmaf(bo, bo, 1.f));   // height of the foot on the outer line
    const float pi = fmaf(bi, rho - ai, z) * frcp(fmaf(bi, bi, 1.f));
    if (no > m && fabsf(po) < dz - m) return kZoneSlant;
    if (ni > m && fabsf(pi) < dz - m) return kZoneSlant + 1;
    if (flags & kFiltVertex) {
        const float zo = copysignf(dz, po), zi = copysignf(dz, pi);
        const float ro = fmaf(bo, zo, ao), ri = fmaf(bi, zi, ai);
        if (fabsf(po) > dz + m && rho > ro + m && ro - fmaf(bi, zo, hole ? ai : 0.f) > 4.f * m)
            return kZoneCorner + (po > 0.f ? 2 : 0);
        if (hole && fabsf(pi) > dz + m && rho < ri - m && fmaf(bo, zi, ao) - ri > 4.f * m)
            return kZoneCorner + 1 + (pi > 0.f ? 2 : 0);
    }
    return kZoneNone;
}

// The zone of a point surely inside the mother: its nearest surface, by 4 delta.
template <class V>
__device__ __forceinline__ int mother_zone(const V& v, const float* p) {
    const float* e = v.m32.e;
    const float d = 4.f * v.m32.delta;
    float s[3];
    int kind[3];
    if (v.m32.kind == KBOX) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s[k] = e[k] - fabsf(p[k]);
            kind[k] = kZonePlane + k;
        }
    } else {
        const float rho = fsqrt(fmaf(p[0], p[0], p[1] * p[1])), az = fabsf(p[2]);
        kind[0] = kZonePlane + 2;
        kind[1] = kZoneOuter;
        kind[2] = kZoneInner;
        if (v.m32.kind == KTUBE) {
            s[0] = e[2] - az;
            s[1] = e[7] - rho;
            s[2] = e[3] != 0.f ? rho - e[8] : f_inf();
        } else {
            s[0] = e[0] - az;
            s[1] = (fmaf(e[2], p[2], e[1]) - rho) * frsqrt(fmaf(e[2], e[2], 1.f));
            s[2] = e[5] != 0.f ? (rho - fmaf(e[4], p[2], e[3])) * frsqrt(fmaf(e[4], e[4], 1.f)) : f_inf();
        }
    }
    float a = s[0], b = f_inf();
    int z = kind[0];
#pragma unroll
    for (int k = 1; k < 3; ++k) {
        const bool first = s[k] < a;
        b = first ? a : fminf(b, s[k]);
        z = first ? kind[k] : z;
        a = fminf(a, s[k]);
    }
    return a > d && a + d < b ? z : kZoneNone;
}

// The FP64 distance of a point in a certain zone of solid r (mother: from
// inside).  Plane zones form one local coordinate; the others share their
// square roots.
__device__ __forceinline__ double zone64(const ShapeRec64& r, int zone, bool mother, double px, double py, double pz) {
    const double* d = r.d;
    const bool plane = zone >= kZonePlane && zone < kZonePlane + 3;
    const int k = plane ? zone - kZonePlane : 0;
    const double w0 = SUB(px, r.t[0]), w1 = SUB(py, r.t[1]), w2 = SUB(pz, r.t[2]);
    double xk, x1 = w1, x2 = w2;
    if (r.flags & kRec64Identity) {
        xk = k == 0 ? w0 : (k == 1 ? w1 : w2);
    } else {
        xk = FMA(r.R[6 + k], w2, FMA(r.R[3 + k], w1, MUL(r.R[k], w0)));
        if (!plane) {
            x1 = FMA(r.R[7], w2, FMA(r.R[4], w1, MUL(r.R[1], w0)));
            x2 = FMA(r.R[8], w2, FMA(r.R[5], w1, MUL(r.R[2], w0)));
        }
    }
    if (plane) {
        const double h = r.kind == KBOX ? d[k] : (r.kind == KTUBE ? d[2] : d[0]);
        const double s = SUB(fabs(xk), h);
        return mother ? -s : s;
    }
    double a, b = 0.0, c;
    if (r.kind == KBOX) {
        a = fmax(SUB(fabs(xk), d[0]), 0.0);
        b = fmax(SUB(fabs(x1), d[1]), 0.0);
        c = fmax(SUB(fabs(x2), d[2]), 0.0);
    } else {
        const double rho = SQRT(DOT2(xk, xk, x1, x1));
        if (zone <= kZoneInner) {
            const bool inner = zone == kZoneInner;
            if (r.kind == KTUBE) {
                const double s = SUB(rho, inner ? d[0] : d[1]);   // outside the outer, in the hole: < 0
                return mother != inner ? -s : s;
            }
            const double s = SUB(FMA(inner ? d[4] : d[2], x2, inner ? d[3] : d[1]), rho);   // the mother cone's
            return MUL(inner ? -s : s, inner ? d[10] : d[9]);
        }
        if (r.kind == KTUBE) {
            a = SUB(fabs(x2), d[2]);
            c = SUB(rho, zone == kZoneCorner ? d[1] : d[0]);
        } else {
            const double dz = d[0];
            const bool inner = zone < kZoneSlant ? ((zone - kZoneCorner) & 1) != 0 : zone == kZoneSlant + 1;
            const double r1 = inner ? r.p[1] : r.p[2], r2 = inner ? r.p[3] : r.p[4];
            if (zone < kZoneSlant) {   // a vertex
                const bool top = (zone - kZoneCorner) >= 2;
                a = SUB(top ? r2 : r1, rho);
                c = SUB(top ? dz : -dz, x2);
            } else {   // seg2 of the outer edge (-dz to +dz) or the inner one (+dz to -dz)
                const double ax = inner ? r2 : r1, az = inner ? dz : -dz, bx = inner ? r1 : r2, bz = inner ? -dz : dz;
                const double ex = SUB(bx, ax), ez = SUB(bz, az);
                const double l2 = DOT2(ex, ex, ez, ez);
                const double f = DIV(DOT2(SUB(rho, ax), ex, SUB(x2, az), ez), l2);
                a = SUB(FMA(f, ex, ax), rho);
                c = SUB(FMA(f, ez, az), x2);
            }
        }
    }
    return SQRT(FMA(a, a, FMA(b, b, MUL(c, c))));
}

// FP64 work of a zone: 0 a plane, 1 one square root, 2 edges and corners, 3 a
// whole solid.
constexpr int kZoneSorts = 4;
__device__ __forceinline__ int zone_sort(int zone) {
    return zone == kZoneNone ? 3 : (zone < kZoneOuter ? 0 : (zone <= kZoneInner ? 1 : 2));
}

// The three least bounds of a point (k: entry of the filter's tables, -1 the mother).
struct Nearest {
    float L1, L2, L3;
    int k1, k2;
};
__device__ __forceinline__ void nearer(Nearest& n, float l, int k) {
    const bool p1 = l < n.L1, p2 = l < n.L2;
    n.L3 = fminf(n.L3, fmaxf(n.L2, l));
    n.k2 = p1 ? n.k1 : (p2 ? k : n.k2);
    n.L2 = fminf(n.L2, fmaxf(n.L1, l));
    n.k1 = p1 ? k : n.k1;
    n.L1 = fminf(n.L1, l);
}

// squared distances of the point to the centres of a FiltSph pair
__device__ __forceinline__ F2 pair_dist2(const float4 a, const float4 b, const F2* p) {
    const F2 w0 = add2(p[0], f2(a.x, a.y)), w1 = add2(p[1], f2(a.z, a.w)), w2 = add2(p[2], f2(b.x, b.y));
    return fma2(w0, w0, fma2(w1, w1, mul2(w2, w2)));
}

// The lowest-index daughter that holds the point of the mother, -1 if none.  `exact(j)`: the FP64 test.
template <class Exact>
__device__ __forceinline__ int point_contains(const FiltTab& f, const float* p, Exact exact) {
    int best = 0x7fffffff;
    float rho = 0.f;
    const F2 p2[3] = {f2(p[0], p[0]), f2(p[1], p[1]), f2(p[2], p[2])};
    for (int base = 0; base < f.nf; base += 32) {
        const FiltSph* S = f.sph + base;
        const int cnt = min(32, f.nf - base), n1 = max(0, min(cnt, f.nq1 - base));
        unsigned m = 0;
        int k = 0;
#pragma unroll 2
        for (; k < n1; ++k) {
            const float4 a = S[k].a, b = S[k].b;
            if (a.w != 0.f) {   // warp-uniform: another axis than the solid before
                const float wx = p[0] - a.x, wy = p[1] - a.y;
                rho = fsqrt(fmaf(wx, wx, wy * wy));
            }
            m |= fabsf(p[2] - a.z) <= b.w && rho <= b.y && rho >= b.z ? 1u << k : 0u;
        }
#pragma unroll 2
        for (; k < cnt; k += 2) {
            const float4 a = S[k].a, b = S[k].b;
            float ca, cb;
            f2_parts(pair_dist2(a, b, p2), ca, cb);
            m |= ((ca <= b.z ? 1u : 0u) | (cb <= b.w ? 2u : 0u)) << k;
        }
        while (m) {
            const FiltHvy* h = f.hvy + base + __ffs(m) - 1;
            m &= m - 1;
            const int in = entry_holds(h, p);
            if (in && h->id < best && (in == 1 || exact(h->id))) best = h->id;
        }
    }
    return best == 0x7fffffff ? -1 : best;
}

// The bounds of every daughter, the mother's already in n.
__device__ __forceinline__ void point_nearest(const FiltTab& f, const float* p, Nearest& n) {
    float rho = 0.f;
    const F2 p2[3] = {f2(p[0], p[0]), f2(p[1], p[1]), f2(p[2], p[2])};
    for (int base = 0; base < f.nf; base += 32) {
        const FiltSph* S = f.sph + base;
        const FiltHvy* H = f.hvy + base;
        const int cnt = min(32, f.nf - base), n1 = max(0, min(cnt, f.nq1 - base));
        int k = 0;
        for (; k < n1; ++k) {
            const float4 a = S[k].a;
            if (a.w != 0.f) {   // warp-uniform: another axis than the solid before
                const float wx = p[0] - a.x, wy = p[1] - a.y;
                rho = fsqrt(fmaf(wx, wx, wy * wy));
            }
            // all lanes read the same record
            const float4 h4 = hvy_words(H + k)[4];
            const float bi = H[k].e[4], z = p[2] - a.z, dz = fabsf(z) - h4.x;
            const bool hole = (H[k].flags & kFiltHole) != 0;
            const float so = rho - fmaf(h4.z, z, h4.y), si = hole ? fmaf(bi, z, h4.w) - rho : -1.f;
            float s;
            if (h4.z == 0.f && bi == 0.f) {
                const float dr = fmaxf(fmaxf(so, si), 0.f), d = fmaxf(dz, 0.f);
                s = fsqrt(fmaf(dr, dr, d * d));
            } else {
                s = fmaxf(fmaxf(dz, so * frsqrt(fmaf(h4.z, h4.z, 1.f))), fmaxf(si * frsqrt(fmaf(bi, bi, 1.f)), 0.f));
            }
            if (S[k].b.y >= 0.f) nearer(n, s * (1.f - kSafMargin), base + k);   // (not a filling entry)
        }
        unsigned m = 0;
#pragma unroll 2
        for (; k < cnt; k += 2) {
            const float4 a = S[k].a, b = S[k].b, c = S[k + 1].a;
            float ca, cb;
            f2_parts(pair_dist2(a, b, p2), ca, cb);
            // distance to the sphere; a filling entry has brad^2 = -1
            const float la = fmaf(fsqrt(ca), 1.f - kSafMargin, -c.x), lb = fmaf(fsqrt(cb), 1.f - kSafMargin, -c.y);
            const bool na = la < n.L2 && b.z > 0.f, nb = lb < n.L2 && b.w > 0.f;
            n.L3 = fminf(n.L3, fminf(na || !(b.z > 0.f) ? f_inf() : la, nb || !(b.w > 0.f) ? f_inf() : lb));
            m |= ((na ? 1u : 0u) | (nb ? 2u : 0u)) << k;
        }
        while (m) {
            const int q = __ffs(m) - 1;
            m &= m - 1;
            nearer(n, entry_distance(H + q, p), base + q);
        }
    }
}

}  // namespace geonav
