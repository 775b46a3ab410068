// filter_pass.cuh -- the FP32 pass of the filter over every daughter of a
// volume, for one track per lane.
//
// What bounds it: issue slots.  A solid's FP32 entry bound costs 45 to 110
// instructions, and a warp that walks the daughters together pays for it
// whenever one lane's track comes near the solid: in the 40-daughter toy
// detector 17 bounds per warp served 2 tracks' worth of candidates each, in
// volumes of many small solids (4 to 200 in cells) 8 to 18 bounds per warp
// served 0.2 to 0.6 candidates per track.  So the pass is split:
//  * a cheap conservative test of every daughter, the same for all lanes and
//    free of branches, sets a bit in the lane's mask (32 daughters at a time);
//  * every lane then walks its OWN bits and bounds its own daughters: one
//    iteration bounds up to 32 different solids, so a warp runs as many as its
//    busiest lane has (about 2 to 4), not the union of its lanes' lists.
// The solids' records are gathered per lane, so they have a layout of their
// own (FiltSph, FiltHvy in geo_internal.h): 16-byte loads, a record stride of
// 112 bytes so that the lanes' gathers from shared memory fall into different
// banks, tubes and cones in one form (a tube is a cone of slope 0) so that
// all quadric solids share one path, daughters sorted by class (unrotated
// quadrics, rotated quadrics, boxes).
//
// The cheap test of boxes and rotated quadrics is the bounding sphere's.  The
// sphere of a long shell or of a flat endcap says little, so an unrotated tube
// or cone gets a lower bound of its entry from its bounding annulus instead:
// the later of reaching its z-slab and its radial range, and a rejection when
// the line misses the outer cylinder, leaves the slab first or moves away
// (2.1 candidates per track pass in the toy detector, of 16; the spheres let
// 8.3 pass).  The lane bounds the solid with the least such value first; when
// that solid is surely entered (below), nothing that starts after the latest
// point of that entry is bounded any more.
//
// Surely entered surfaces.  An FP64 instruction holds its unit for 64 cycles
// per warp, and DistFromOutside tries every surface of a solid, each quadric
// with a square root and a division.  So the bound also says which surface the
// exact line enters through, when that is certain, and FP64 evaluates that
// surface alone, with the same operations as the whole routine and so the
// same bits (surface64 in nav_refine.cuh).  The premise is that of the
// inflation, with the room it leaves: the FP32 line lies within delta / 2 of
// the exact one, rounding of the quadrics included (48 eps32 S of the
// extent S are in delta; the roundings of position, direction, shift and
// rotation add up to less than 16).  The copy is delta larger than the solid,
// so the exact crossing is that of a solid delta / 2 to 3 delta / 2 smaller
// than the copy.  Certain then means: under such a change the crossing lies in
// [t, t + e]; over that interval it keeps clear of every limit of its
// acceptance (no edge nearby); no other surface of the solid has a crossing before
// t + e; and the start is outside the inflated copy.  e is 2 delta / |u_z| for
// an end plane and 2 delta R / sqrt(D) for a quadric (R / sqrt(D) is the
// crossing's derivative by R), used only where D exceeds four times its own
// change.  An accepted crossing that keeps clear of the edges is the
// entry: before it the line is outside the surface's constraint, which every
// earlier entry would have to satisfy.  The upper bound t + e of a certain
// entry is also what the cut above uses.
#pragma once
#include "geo_internal.h"
#include "shapes32.cuh"

namespace geonav {

// Candidates kept per track: the kCand smallest FP32 bounds, and the least
// bound evicted.  Two suffice: on every test scene, random and adversarial
// rays, no track falls back to the full FP64 loop, and the list's registers
// and insertion work are what the FP32 pass can least afford.
constexpr int kCand = 2;

// A candidate is its daughter's index and, from bit kTagShift on, the surface it
// is surely entered through (kTagNone: not certain).
constexpr int kTagShift = 24;
constexpr int kIdMask = (1 << kTagShift) - 1;
enum : int { kTagNone = 0, kTagPlane = 1, kTagOuter = 2, kTagInner = 3, kTagAxis = 4 };   // kTagAxis + k: a box's axis k

struct Cands {
    float L[kCand];
    int j[kCand];
    int n;
    float dropped;   // smallest bound evicted from the list
};

__device__ __forceinline__ void cands_clear(Cands& c) {
#pragma unroll
    for (int k = 0; k < kCand; ++k) {
        c.L[k] = f_inf();
        c.j[k] = 0;
    }
    c.n = 0;
    c.dropped = f_inf();
}

// whether the list holds daughter j
__device__ __forceinline__ bool cand_holds(const Cands& c, int j) {
    return (c.L[0] < f_inf() && (c.j[0] & kIdMask) == j) || (c.L[1] < f_inf() && (c.j[1] & kIdMask) == j);
}

// Insertion of a finite bound.  An empty slot holds +inf, so no count is needed: the
// list's n is its number of finite bounds (cands_count).
__device__ __forceinline__ void cand_put(Cands& c, float L, int j) {
    static_assert(kCand == 2, "written out for a list of two");
    c.dropped = fminf(c.dropped, fmaxf(L, c.L[1]));
    const bool p0 = L < c.L[0], p1 = L < c.L[1];
    c.j[1] = p0 ? c.j[0] : (p1 ? j : c.j[1]);
    c.L[1] = p0 ? c.L[0] : fminf(L, c.L[1]);
    c.j[0] = p0 ? j : c.j[0];
    c.L[0] = fminf(L, c.L[0]);
}
__device__ __forceinline__ void cands_count(Cands& c) {
    c.n = (c.L[0] < f_inf() ? 1 : 0) + (c.L[1] < f_inf() ? 1 : 0);
}

// lower the FP32 parameter t by its rounding allowance
__device__ __forceinline__ float lower_bound(float t, float delta, float inv_dn) {
    return t - (16.f * kEps32f * fabsf(t) + delta * inv_dn);
}

// The FP32 track: position, direction, e = -d / |d|^2 (the shift to the closest
// approach is w . e), 1 / |d| rounded up.
struct Ray32 {
    float p[3], d[3], e[3];
    float inv_dn;
};

struct FiltTab {
    const FiltSph* sph;
    const FiltHvy* hvy;
    int nq1, nq, nf;   // unrotated quadrics [0, nq1), rotated [nq1, nq), boxes [nq, nf)
};

__device__ __forceinline__ void to_shifted(const float4 h0, const Ray32& r, float& s0, float* q) {
    const float w0 = r.p[0] - h0.x, w1 = r.p[1] - h0.y, w2 = r.p[2] - h0.z;
    s0 = fmaf(w0, r.e[0], fmaf(w1, r.e[1], w2 * r.e[2]));
    q[0] = fmaf(s0, r.d[0], w0);
    q[1] = fmaf(s0, r.d[1], w1);
    q[2] = fmaf(s0, r.d[2], w2);
}

// R^T a for the record's rotation (h1, h2, h3.x: row-major local -> mother)
__device__ __forceinline__ void rotate_in(const float4 h1, const float4 h2, const float r8, const float* a, float* x) {
    x[0] = fmaf(h2.z, a[2], fmaf(h1.w, a[1], h1.x * a[0]));
    x[1] = fmaf(h2.w, a[2], fmaf(h2.x, a[1], h1.y * a[0]));
    x[2] = fmaf(r8, a[2], fmaf(h2.y, a[1], h1.z * a[0]));
}

__device__ __forceinline__ const float4* hvy_words(const FiltHvy* h) { return reinterpret_cast<const float4*>(h); }

// Bound of the entry into quadric solid h (tube or cone; cone_enter32's),
// inserted into the list when it is within Um.  Returns the latest parameter of
// a certain entry, else +inf.
__device__ __forceinline__ float bound_quad(const FiltHvy* h, const Ray32& r, float Um, Cands& c) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h3 = H[3], h4 = H[4], h5 = H[5], h6 = H[6];
    const float tol = h6.z;
    const int flags = __float_as_int(h3.y);
    float s0, x[3], u[3];
    to_shifted(h0, r, s0, x);
    u[0] = r.d[0]; u[1] = r.d[1]; u[2] = r.d[2];
    if (!(flags & kFiltIdentity)) {
        const float4 h1 = H[1], h2 = H[2];
        const float q[3] = {x[0], x[1], x[2]};
        rotate_in(h1, h2, h3.x, q, x);
        rotate_in(h1, h2, h3.x, r.d, u);
    }
    const bool hole = (flags & kFiltHole) != 0;
    const float dz = h4.x, ao = h4.y, bo = h4.z, ai = h4.w, bi = h5.x, zl = h3.w;
    const float tmin = -s0;
    const float sx = fmaf(tmin, u[0], x[0]), sy = fmaf(tmin, u[1], x[1]), sz = fmaf(tmin, u[2], x[2]);
    const float sr2 = fmaf(sx, sx, sy * sy);
    const float ro = fmaf(bo, sz, ao) + tol, ri = fmaf(bi, sz, ai) - tol;
    const bool in0 = fabsf(sz) <= zl && sr2 <= ro * ro && (!hole || ri <= 0.f || sr2 >= ri * ri);
    const float A0 = fmaf(u[0], u[0], u[1] * u[1]);
    const float B0 = fmaf(x[0], u[0], x[1] * u[1]);
    const float rho2 = fmaf(x[0], x[0], x[1] * x[1]);
    const float tol2 = 2.f * tol, az = fabsf(u[2]);
    float best, e, second = f_inf();
    int tag = kTagPlane;
    bool sure;
    {   // the end plane the start lies beyond, when the track approaches it
        const float inv = fdiv(1.f, u[2]);
        const float ze = copysignf(dz, sz);
        const float tz = (ze - x[2]) * inv;
        const float xh = fmaf(tz, u[0], x[0]), yh = fmaf(tz, u[1], x[1]);
        const float r2 = fmaf(xh, xh, yh * yh);
        const bool up = sz > 0.f;
        const float hi2 = up ? h5.z : h5.y, lo2 = up ? h6.x : h5.w;
        best = fabsf(sz) > dz && sz * u[2] < 0.f && r2 <= hi2 && r2 >= lo2 ? fmaxf(tz, tmin) : f_inf();
        e = tol2 * fabsf(inv);
        // against the solid's own annulus: its radius lines at its own end (the
        // copy's are delta sqrt(1 + slope^2) further out, and its end delta)
        const float rh = fsqrt(r2), slack = fmaf(e, fsqrt(A0), fmaf(0.5f, h6.y, tol)), zt = copysignf(dz - tol, sz);
        sure = rh + slack <= fmaf(bo, zt, ao) && (!hole || rh - slack >= fmaf(bi, zt, ai));
    }
    const float zs = dz - tol2;
    auto quadric = [&](float a, float b, bool rising, int its) {
        const float r0 = fmaf(b, x[2], a), rs = b * u[2];
        const float A = fmaf(-rs, rs, A0), B = fmaf(-r0, rs, B0), C = fmaf(-r0, r0, rho2);
        // the falling root of the quadric, or (its signs turned) the rising one
        const float sg = rising ? -1.f : 1.f;
        float sq;
        const bool real = disc32(A, B, C, sq);
        const float Bs = sg * B;
        const bool bneg = Bs < 0.f;
        const float s0r = fdiv(bneg ? sg * C : -Bs - sq, bneg ? sq - Bs : sg * A);
        const float s = real && (bneg || A != 0.f) ? s0r : f_inf();
        const float z = fmaf(s, u[2], x[2]);
        if (s >= tmin && fabsf(z) <= zl) {
            const float es = fdiv(h6.y * fabsf(fmaf(s, rs, r0)), sq);   // h6.y: 2 delta sqrt(1 + slope^2)
            const bool ok = sq * sq > 6.f * h6.y * fmaf(A0, h6.y, fabsf(fmaf(A, r0, -B * rs))) &&
                            fmaf(az, es, fabsf(z)) <= zs;
            const bool first = s < best;
            second = first ? best : fminf(second, s);
            e = first ? es : e;
            sure = first ? ok : sure;
            tag = first ? its : tag;
            best = fminf(best, s);
        }
    };
    quadric(ao, bo, false, kTagOuter);
    if (hole) quadric(ai, bi, true, kTagInner);
    best = in0 ? tmin : best;
    const float L = lower_bound(s0 + best, tol, r.inv_dn);
    if (!(best < f_inf() && L <= Um)) return f_inf();
    const float last = best + e;
    sure = sure && !in0 && !(flags & kFiltLoose) && last + 32.f * kEps32f * fabsf(last) < second;
    cand_put(c, L, __float_as_int(h3.z) | (sure ? tag << kTagShift : 0));
    return sure ? fmaf(32.f * kEps32f, fabsf(s0 + last), s0 + last) + tol2 * r.inv_dn : f_inf();
}

// The same for a box: the axis of the latest slab entry, certain when it stays
// the latest, and before every slab's exit, under a change of 2 delta.
__device__ __forceinline__ float bound_box(const FiltHvy* h, const Ray32& r, float Um, Cands& c) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h1 = H[1], h2 = H[2], h3 = H[3], h4 = H[4];
    const float tol = h4.w;
    float s0, q[3], x[3], u[3];
    to_shifted(h0, r, s0, q);
    rotate_in(h1, h2, h3.x, q, x);
    rotate_in(h1, h2, h3.x, r.d, u);
    const float hh[3] = {h4.x, h4.y, h4.z};
    const float tmin = -s0;
    float tn = tmin, tf = f_inf();           // the entry, and the least exit
    float last = -f_inf(), out = f_inf();    // the latest entry, and the least exit, of the true box
    float others = -f_inf();                 // the latest entry through the axes before the best one, or after it
    int tag = kTagNone;
    float lastk = -f_inf();                  // the best axis's latest entry
    bool miss = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float inv = fdiv(1.f, u[k]);
        const float a0 = (-hh[k] - x[k]) * inv, b0 = (hh[k] - x[k]) * inv;
        const float a = fminf(a0, b0), b = fmaxf(a0, b0);
        const float e = 2.f * tol * fabsf(inv);
        if (u[k] == 0.f) {
            miss = miss || fabsf(x[k]) > hh[k] + tol;
            out = -f_inf();   // not certain
        } else {
            const bool first = a > tn;
            others = fmaxf(others, first ? lastk : a + e);
            lastk = first ? a + e : lastk;
            tag = first ? kTagAxis + k : tag;
            tn = fmaxf(tn, a);
            tf = fminf(tf, b);
            last = fmaxf(last, a + e);
            out = fminf(out, b - e);
        }
    }
    if (miss || !(tn <= tf)) return f_inf();
    const float L = lower_bound(s0 + tn, tol, r.inv_dn);
    if (!(L <= Um)) return f_inf();
    const float m = 32.f * kEps32f * fmaxf(fabsf(tn), fabsf(last));
    const bool sure = tag != kTagNone && tn - m > others && last + m < out && tn > tmin + m + 2.f * tol * r.inv_dn;
    cand_put(c, L, __float_as_int(h3.z) | (sure ? tag << kTagShift : 0));
    return sure ? fmaf(32.f * kEps32f, fabsf(s0 + last), s0 + last) + 2.f * tol * r.inv_dn : f_inf();
}

// Two FP32 values in one register pair: one instruction for both (the
// arithmetic rate is that of two instructions, but the pass is bound by issue
// slots).
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_parts(F2 a, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// The track's values in both halves, for the paired sphere tests.
struct Ray2 {
    F2 p[3], d[3], e[3], inv, ninv;
};
__device__ __forceinline__ Ray2 pair_ray(const Ray32& r) {
    Ray2 q;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        q.p[k] = f2(r.p[k], r.p[k]);
        q.d[k] = f2(r.d[k], r.d[k]);
        q.e[k] = f2(r.e[k], r.e[k]);
    }
    q.inv = f2(r.inv_dn, r.inv_dn);
    q.ninv = f2(-r.inv_dn, -r.inv_dn);
    return q;
}

// Bounding-sphere tests of two daughters (a FiltSph pair): the line passes the
// sphere, ahead of the start and before Um.  Bits 0 and 1.
__device__ __forceinline__ unsigned spheres_ahead(const FiltSph* S, const Ray2& r, float Um) {
    const float4 a = S[0].a, b = S[0].b, c = S[1].a;   // (-tx, -tx, -ty, -ty), (-tz, -tz, brad^2, brad^2), (brad, brad)
    const F2 w0 = add2(r.p[0], f2(a.x, a.y)), w1 = add2(r.p[1], f2(a.z, a.w)), w2 = add2(r.p[2], f2(b.x, b.y));
    const F2 s0 = fma2(w0, r.e[0], fma2(w1, r.e[1], mul2(w2, r.e[2])));
    const F2 q0 = fma2(s0, r.d[0], w0), q1 = fma2(s0, r.d[1], w1), q2 = fma2(s0, r.d[2], w2);
    const F2 perp2 = fma2(q0, q0, fma2(q1, q1, mul2(q2, q2)));
    const F2 rad = f2(c.x, c.y);
    const F2 hi = fma2(rad, r.inv, s0), lo = fma2(rad, r.ninv, s0);
    float pa, pb, ha, hb, la, lb;
    f2_parts(perp2, pa, pb);
    f2_parts(hi, ha, hb);
    f2_parts(lo, la, lb);
    return (pa <= b.z && ha >= 0.f && la <= Um ? 1u : 0u) | (pb <= b.w && hb >= 0.f && lb <= Um ? 2u : 0u);
}

// Annulus test of an unrotated quadric: a lower bound of the entry, +inf when
// the track cannot enter before Um.  The limits (Rmax, Rmin, half-length) are
// those of the inflated copy plus delta; inv_lo and inv_hi are 1 / |u_z| and
// 1 / |u_perp| with a relative margin below and above.
struct AxisRay {
    float rho, crs;      // distance of the start, and of the line, to the axis
    float rr;            // least distance to the axis along the forward ray
};
__device__ __forceinline__ void to_axis(const float4 a, const Ray32& r, float inv_perp, AxisRay& x) {
    const float wx = r.p[0] - a.x, wy = r.p[1] - a.y;
    x.rho = fsqrt(fmaf(wx, wx, wy * wy));
    x.crs = fabsf(fmaf(wx, r.d[1], -(wy * r.d[0]))) * inv_perp;
    x.rr = fmaf(wx, r.d[0], wy * r.d[1]) >= 0.f ? x.rho : x.crs;
}
__device__ __forceinline__ float annulus_bound(const float tz, const float4 b, const AxisRay& x, const Ray32& r,
                                               float inv_z_lo, float inv_z_hi, float inv_r_lo, float Um) {
    const float wz = r.p[2] - tz;
    const float wzs = r.d[2] < 0.f ? -wz : wz;
    const float t_in = (-b.w - wzs) * inv_z_lo, t_out = (b.w - wzs) * inv_z_hi;
    const float t_r = fmaxf(x.rho - b.y, b.z - x.rho) * inv_r_lo;
    const float L = fmaxf(fmaxf(t_in, t_r), 0.f);
    return t_out < L || x.rr > b.y || L > Um ? f_inf() : L;
}

// The uniform grid of a volume as the walk reads it: the short form staged in
// shared memory (cells: offset | count << 16, 16-bit entries) or the CSR lists
// in global memory.
struct GridTab {
    const uint32_t* cells;
    const uint16_t* ids16;
    const int32_t* off;
    const int32_t* fids;
    const FiltHvy* hvy;
};

// The daughters listed in the cells that the track crosses before Um (3D-DDA
// along the FP32 ray; at most gx + gy + gz + 3 cells).  What bounds it: the lanes'
// own walks diverge, so the loop is flat -- every turn a lane goes on to its
// next cell if its list is done, then looks at one entry -- until the lane holds a
// daughter whose sphere it meets; then all lanes bound their daughters
// together.  A certain entry shortens Um and with it the walk (the
// 512-daughter volume: about half of the tracks enter a daughter, most
// far before the mother's exit).  A daughter met again is skipped (4-entry mailbox,
// then the candidate list).
template <bool SMALL>
__device__ __forceinline__ void filter_grid(const VolView& v, const GridTab& g, const Ray32& r, float Um, Cands& c) {
    // per axis: cells left before the walk leaves the grid, stride of the
    // linear index, next boundary parameter, increment
    int n0, n1, n2, s0, s1, s2;
    float m0, m1, m2, e0, e1, e2;
    int cell = 0;
    auto setup = [&](int k, int pitch, int& left, int& st, float& tm, float& te) {
        const float lo = v.lo32[k], w = v.cell32[k];
        const int gk = v.grid[k];
        int ii = int(floorf((r.p[k] - lo) * v.inv_cell32[k]));
        ii = ii < 0 ? 0 : (ii >= gk ? gk - 1 : ii);
        cell += ii * pitch;
        const float d = r.d[k], inv = frcp(d);
        const bool up = d > 0.f;
        st = up ? pitch : -pitch;
        left = up ? gk - 1 - ii : ii;
        tm = d != 0.f ? (fmaf(float(up ? ii + 1 : ii), w, lo) - r.p[k]) * inv : f_inf();
        te = d != 0.f ? w * fabsf(inv) : f_inf();
    };
    setup(0, v.grid[1] * v.grid[2], n0, s0, m0, e0);
    setup(1, v.grid[2], n1, s1, m1, e1);
    setup(2, 1, n2, s2, m2, e2);
    int cur, end;
    auto open = [&] {
        if (SMALL) {
            const uint32_t w = g.cells[cell];
            cur = int(w & 0xffffu);
            end = cur + int(w >> 16);
        } else {
            cur = g.off[cell];
            end = g.off[cell + 1];
        }
    };
    open();
    int mb0 = -1, mb1 = -1, mb2 = -1, mb3 = -1;
    bool more = true;
    while (more) {
        int found = -1;
        do {
            if (cur >= end) {   // the next cell, if the track reaches it before Um
                const float mn = fminf(m0, fminf(m1, m2));
                const bool a0 = m0 <= mn, a1 = !a0 && m1 <= mn, a2 = !a0 && !a1;
                more = mn <= Um && (a0 ? n0 : (a1 ? n1 : n2)) > 0;
                cell += a0 ? s0 : (a1 ? s1 : s2);
                n0 -= a0;
                n1 -= a1;
                n2 -= a2;
                m0 = a0 ? m0 + e0 : m0;
                m1 = a1 ? m1 + e1 : m1;
                m2 = a2 ? m2 + e2 : m2;
                if (more) open();
            }
            if (cur < end) {   // the next entry of its list
                const int j = SMALL ? int(g.ids16[cur]) : g.fids[cur];
                ++cur;
                if (j != mb0 && j != mb1 && j != mb2 && j != mb3) {
                    mb3 = mb2; mb2 = mb1; mb1 = mb0; mb0 = j;
                    const float4 h0 = hvy_words(g.hvy + j)[0];
                    float t0, q[3];
                    to_shifted(h0, r, t0, q);
                    const float perp2 = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2]));
                    const float half = h0.w * r.inv_dn;
                    if (perp2 <= h0.w * h0.w * (1.f + 4.f * kEps32f) && t0 >= -half && t0 - half <= Um) found = j;
                }
            }
        } while (found < 0 && more);
        if (found >= 0) {
            const FiltHvy* h = g.hvy + found;
            if (!cand_holds(c, h->id))
                Um = fminf(Um, (h->flags & kFiltBox) ? bound_box(h, r, Um, c) : bound_quad(h, r, Um, c));
        }
    }
    cands_count(c);
}

// Re-entry of a track into solid h that it has just left (it starts on the
// solid's surface): kReentryNone when the exact line surely does not enter it again,
// the surface (kTagOuter / kTagInner) of the sure next entry with a lower
// bound of its parameter in L, kTagNone when it is not certain.  The margins
// are those of a certain entry (above).
constexpr int kReentryNone = -1;
__device__ __forceinline__ int reentry32(const FiltHvy* h, const Ray32& r, float& L) {
    const float4* H = hvy_words(h);
    const float4 h0 = H[0], h3 = H[3], h4 = H[4];
    const int flags = __float_as_int(h3.y);
    L = 0.f;
    if (flags & kFiltLoose) return kTagNone;
    const float w[3] = {r.p[0] - h0.x, r.p[1] - h0.y, r.p[2] - h0.z};
    float x[3], u[3];
    if (flags & kFiltIdentity) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = w[k];
            u[k] = r.d[k];
        }
    } else {
        const float4 h1 = H[1], h2 = H[2];
        rotate_in(h1, h2, h3.x, w, x);
        rotate_in(h1, h2, h3.x, r.d, u);
    }
    const float umin = 16.f * kEps32f * frcp(r.inv_dn);   // a component's sign is certain above it
    if (flags & kFiltBox) {
        // one face near, the track moving out of its slab, the others far: the
        // box's exit from that slab lies behind the start
        const float d = h4.w, hh[3] = {h4.x, h4.y, h4.z};
        int near = 0;
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float a = fabsf(x[k]) - (hh[k] - d);
            if (a > -2.f * d) {
                ++near;
                ok = ok && a < 2.f * d && fabsf(x[k]) > 2.f * d && x[k] * u[k] > 0.f && fabsf(u[k]) > umin;
            }
        }
        return ok && near == 1 ? kReentryNone : kTagNone;
    }
    const float4 h5 = H[5], h6 = H[6];
    const float d = h6.z, g = h6.y, dz = h4.x - d;
    const float az = fabsf(x[2]) - dz;
    if (az > 2.f * d || (az > -2.f * d && !(fabsf(x[2]) > 2.f * d && x[2] * u[2] > 0.f && fabsf(u[2]) > umin)))
        return kTagNone;
    const float A0 = fmaf(u[0], u[0], u[1] * u[1]);
    const float B0 = fmaf(x[0], u[0], x[1] * u[1]);
    const float rho2 = fmaf(x[0], x[0], x[1] * x[1]);
    float hi = f_inf();   // the entry found lies in [L, hi]
    int tag = kReentryNone;
    bool ok = true;
    // (the copy's radius lines: the solid's own are delta away, inside g's margin)
    auto quadric = [&](float a, float b, bool rising, int its) {
        const float r0 = fmaf(b, x[2], a), rs = b * u[2];
        const float A = fmaf(-rs, rs, A0), B = fmaf(-r0, rs, B0), C = fmaf(-r0, r0, rho2);
        const float D = fmaf(B, B, -A * C);
        const float change = 6.f * g * fmaf(A0, g, fabsf(fmaf(A, r0, -B * rs)));
        if (D < -change - 16.f * kEps32f * fmaf(B, B, fabsf(A * C))) return;   // no crossing at all
        if (!(D > change) || !(fabsf(A) > 1e-6f * A0)) {
            ok = false;
            return;
        }
        const float sq = fsqrt(D), sg = rising ? -1.f : 1.f, Bs = sg * B;
        const bool bneg = Bs < 0.f;
        const float s = fdiv(bneg ? sg * C : -Bs - sq, bneg ? sq - Bs : sg * A);
        const float e = fmaf(32.f * kEps32f, fabsf(s), fdiv(g * fabsf(fmaf(s, rs, r0)), sq)) + 2.f * d * r.inv_dn;
        if (s < -e || s - e > hi) return;   // behind, or after the other entry
        const float z = fabsf(fmaf(s, u[2], x[2])), zs = fmaf(fabsf(u[2]), e, 2.f * d);
        if (s > e && z - zs > dz) return;   // beyond the ends
        const bool sure = s > e && z + zs < dz;
        ok = ok && sure && (tag == kReentryNone || s + e < L);
        hi = s + e;
        L = s - e;
        tag = its;
    };
    quadric(h4.y, h4.z, false, kTagOuter);
    if (ok && (flags & kFiltHole)) quadric(h4.w, h5.x, true, kTagInner);
    return ok ? tag : kTagNone;
}

// Every daughter of the volume, 32 at a time: the cheap tests together, then
// each lane's own solids (one call site per kind of bound: the pass's code has
// to stay small, warps run its parts at different times and share the
// instruction caches).
// SKIP: the entry `skip` (-1 none) is left out.
template <bool SKIP = false>
__device__ __forceinline__ void filter_daughters(const FiltTab& f, const Ray32& r, float Um, Cands& c, int skip = -1) {
    // a direction within 1e-6 of the axis: no radial bound (its FP32
    // perpendicular part may have lost its precision)
    const float perp2 = fmaf(r.d[0], r.d[0], r.d[1] * r.d[1]);
    const float inv_z = frcp(fabsf(r.d[2]));
    const float inv_r = perp2 > 1e-12f * fmaf(r.d[2], r.d[2], perp2) ? frsqrt(perp2) : 0.f;
    const float inv_z_lo = inv_z * (1.f - 16.f * kEps32f), inv_z_hi = inv_z * (1.f + 32.f * kEps32f);
    const float inv_r_lo = inv_r * (1.f - 16.f * kEps32f);
    AxisRay ax = {0.f, 0.f, 0.f};
    for (int base = 0; base < f.nf; base += 32) {
        const FiltSph* S = f.sph + base;
        const FiltHvy* H = f.hvy + base;
        const int cnt = min(32, f.nf - base), n1 = max(0, min(cnt, f.nq1 - base)), n2 = max(0, min(cnt, f.nq - base));
        unsigned m = 0;                       // the lane's solids: annulus bits, sphere bits
        float l1 = f_inf(), l2 = f_inf(), l3 = f_inf();   // the least annulus bounds
        int k1 = -1, k2 = -1, k = 0;
#pragma unroll 2
        for (; k < n1; ++k) {
            const float4 a = S[k].a, b = S[k].b;
            if (a.w != 0.f) to_axis(a, r, inv_r, ax);   // warp-uniform: another axis than the solid before
            float L = annulus_bound(a.z, b, ax, r, inv_z_lo, inv_z_hi, inv_r_lo, Um);
            if (SKIP) L = base + k == skip ? f_inf() : L;
            m |= L < f_inf() ? 1u << k : 0u;
            const bool p1 = L < l1, p2 = L < l2;
            l3 = fminf(l3, fmaxf(l2, L));
            k2 = p1 ? k1 : (p2 ? k : k2);
            l2 = fminf(l2, fmaxf(l1, L));
            k1 = p1 ? k : k1;
            l1 = fminf(l1, L);
        }
        if (n1 < cnt) {
            const Ray2 r2 = pair_ray(r);
            k = n1;
#pragma unroll 2
            for (; k < cnt; k += 2) m |= spheres_ahead(S + k, r2, Um) << k;
        }
        if (SKIP && skip >= base && skip < base + 32) m &= ~(1u << (skip - base));
        // quadrics: the two with the least annulus bounds first, then the
        // others in order; an annulus bit is looked at again, against the bound
        // Um of what has been found since
        const unsigned quads = n2 >= 32 ? 0xffffffffu : (1u << n2) - 1u;
        const unsigned later = n1 >= 32 ? 0u : ~((1u << n1) - 1u);   // the bits that are no annuli
        unsigned mq = m & quads;
        if (k1 >= 0) mq &= ~(1u << k1);
        if (k2 >= 0) mq &= ~(1u << k2);
        for (;;) {
            int q = k1;
            if (q < 0) {
                if (l3 > Um) mq &= later;   // no other annulus starts before Um
                while (mq) {
                    const int w = __ffs(mq) - 1;
                    mq &= mq - 1;
                    q = w;
                    if (w >= n1) break;
                    const float4 a = S[w].a, b = S[w].b;
                    AxisRay aq;
                    to_axis(a, r, inv_r, aq);
                    if (annulus_bound(a.z, b, aq, r, inv_z_lo, inv_z_hi, inv_r_lo, Um) < f_inf()) break;
                    q = -1;
                }
            }
            if (q < 0) break;
            Um = fminf(Um, bound_quad(H + q, r, Um, c));
            k1 = l2 <= Um ? k2 : -1;
            k2 = -1;
        }
        unsigned mb = m & ~quads;
        while (mb) {
            const int q = __ffs(mb) - 1;
            mb &= mb - 1;
            Um = fminf(Um, bound_box(H + q, r, Um, c));
        }
    }
    cands_count(c);
}

}  // namespace geonav
