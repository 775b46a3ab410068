// nav_refine.cuh -- per-track step of the FP32-filter + FP64-refine
// navigator (see nav_refine.cu for the scheme).  Shared by every kernel that
// navigates with the filter.
#pragma once
#include "filter_pass.cuh"
#include "geo_internal.h"
#include "nav_common.cuh"
#include "shapes32.cuh"
#include "shapes64.cuh"

namespace geonav {

// FP32 lower bound of one daughter's DistFromOutside (bounding-sphere test,
// transform in the frame shifted to the closest approach, inflated solid),
// inserted into the candidate list when it can beat the mother's exit.  For
// lanes that visit the same daughter together.
__device__ __forceinline__ void bound_daughter(const ShapeRec32& r, int j, const Ray32& ray, float Um, Cands& c) {
    const float4 tb = *reinterpret_cast<const float4*>(r.t);   // t and brad^2
    float s0, q[3];
    to_shifted(tb, ray, s0, q);
    const float perp2 = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2]));
    if (perp2 > tb.w) return;
    const float half = r.brad * ray.inv_dn;
    if (s0 + half < 0.f || s0 - half > Um) return;
    float x[3], u[3];
    if (r.flags & kRec32Identity) {   // warp-uniform: every lane visits solid j together
        x[0] = q[0]; x[1] = q[1]; x[2] = q[2];
        u[0] = ray.d[0]; u[1] = ray.d[1]; u[2] = ray.d[2];
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = fmaf(r.R[6 + k], q[2], fmaf(r.R[3 + k], q[1], r.R[k] * q[0]));
            u[k] = fmaf(r.R[6 + k], ray.d[2], fmaf(r.R[3 + k], ray.d[1], r.R[k] * ray.d[0]));
        }
    }
    const float tp = enter32(r, x, u, -s0);
    if (!(tp < f_inf())) return;
    const float L = lower_bound(s0 + tp, r.delta, ray.inv_dn);
    if (L > Um) return;
    cand_put(c, L, j);
}

// The filter's cold FP64 paths (a direction magnitude outside the FP32
// range, a start between the mother's shrunk copy and the mother, a bound
// evicted from the list that could still win), out of line: inlined, their
// FP64 code raised the register pressure of the hot FP32 pass (spill stores
// 400 -> 148 bytes; toy detector 0.2268 -> 0.2237 ms, the batched launch
// 1.128 -> 1.106 ms).
template <bool SEGS>
static __device__ __noinline__ void nav_all64_cold(const ShapeRec64& m, const ShapeRec64* __restrict__ tab, int nd,
                                                   double px, double py, double pz, double qx, double qy, double qz,
                                                   double& best, int& h) {
    nav_all64<SEGS>(m, tab, nd, px, py, pz, qx, qy, qz, best, h);
}
template <bool SEGS>
static __device__ __noinline__ bool contains64_cold(const ShapeRec64& m, double px, double py, double pz) {
    const double p[3] = {px, py, pz};
    return contains64<SEGS>(m, p);
}

// State of one track between the FP32 pass and the FP64 refinement.
struct RefineState {
    Cands c;
    float Lm;       // lower bound of the mother's exit
    int tag;        // the surface the first task is surely decided by (kTagNone: not certain)
    int status;     // 0: refine, 1: result already final (invalid / outside / fallback)
};

// The first solid to refine: the mother (-1) when its bound comes first or
// there is no candidate, else candidate 0.
__device__ __forceinline__ int first_task(const RefineState& st) {
    return (st.c.n == 0 || st.Lm <= st.c.L[0]) ? -1 : st.c.j[0];
}

// The mother's exit: the shrunk copy gives "surely inside" and a lower bound,
// the grown copy an upper bound, and both together the surface the exact exit
// crosses when that is certain: its exit from the grown copy comes before every
// other surface's exit from the shrunk one.
struct MotherExit {
    float lo, hi;
    bool in;    // inside the shrunk copy: the bounds hold
    int tag;    // kTagPlane / kTagOuter / kTagInner, a box's kTagAxis + k, kTagNone: not certain
};

// `entered`: the track starts on the mother's surface, moving in.  The bounds
// hold then as well (`in`) when the line crosses the shrunk copy's outer
// surface (it does not graze it) and does not leave through the inner one at
// its start: it starts off that surface, or moves away from the axis.
// A hole bounds the exit from above only for starts surely off its surface.  On
// it, FP64 may find its crossing a rounding behind the start and pass over it
// (a cone's, or any entered mother's), so that the exact exit is the next one,
// beyond the hole.
// V holds the solid's copies m32 (shrunk), m32u (grown) and its record m64.
template <bool ENTERED = false, class V>
__device__ __forceinline__ MotherExit mother_exit32(const V& v, const Ray32& r, bool entered = false) {
    const float *el = v.m32.e, *eh = v.m32u.e, *x = r.p, *u = r.d;
    MotherExit m;
    float second = f_inf(), thi = f_inf();
    bool crosses = true;   // (entered)
    m.lo = m.hi = f_inf();
    m.tag = kTagNone;
    auto take = [&](float lo, float hi, int tag) {
        const bool first = lo < m.lo;
        second = first ? m.lo : fminf(second, lo);
        m.tag = first ? tag : m.tag;
        thi = first ? hi : thi;
        m.lo = fminf(m.lo, lo);
        m.hi = fminf(m.hi, hi);
    };
    auto plane = [&](int k, float hl, float hh, int tag) {
        if (u[k] != 0.f) take(fdiv(copysignf(hl, u[k]) - x[k], u[k]), fdiv(copysignf(hh, u[k]) - x[k], u[k]), tag);
    };
    const int kind = v.m32.kind;
    if (kind == KBOX) {
        m.in = fabsf(x[0]) <= el[0] && fabsf(x[1]) <= el[1] && fabsf(x[2]) <= el[2];
#pragma unroll
        for (int k = 0; k < 3; ++k) plane(k, el[k], eh[k], kTagAxis + k);
    } else {
        const float rho2 = fmaf(x[0], x[0], x[1] * x[1]);
        const float A0 = fmaf(u[0], u[0], u[1] * u[1]);
        const float B0 = fmaf(x[0], u[0], x[1] * u[1]);
        // both copies' quadrics: the outer one left where it rises, the inner one where it falls
        auto outer = [&](float Al, float Bl, float Cl, float Ah, float Bh, float Ch) {
            const float lo = root_rising32(Al, Bl, Cl), hi = root_rising32(Ah, Bh, Ch);
            if (ENTERED) crosses = fmaf(Bl, Bl, -Al * Cl) > 16.f * kEps32f * fmaf(Bl, Bl, fabsf(Al * Cl)) && lo >= 0.f;
            take(lo >= 0.f ? lo : f_inf(), hi >= 0.f ? hi : f_inf(), kTagOuter);
        };
        auto inner = [&](float Al, float Bl, float Cl, bool hole, float Ah, float Bh, float Ch) {
            const float lo = root_falling32(Al, Bl, Cl), hi = hole ? root_falling32(Ah, Bh, Ch) : f_inf();
            if (ENTERED) crosses = crosses && (Cl >= 0.f || Bl > 64.f * kEps32f * fsqrt(Al > 0.f ? Al * rho2 : f_inf()));
            const bool off = Cl >= 0.f || (ENTERED && entered && crosses);
            take(lo >= 0.f ? lo : f_inf(), off && hi >= 0.f ? hi : f_inf(), kTagInner);
        };
        if (kind == KTUBE) {
            m.in = fabsf(x[2]) <= el[2] && rho2 <= el[1] && (el[3] == 0.f || rho2 >= el[0]);
            plane(2, el[2], eh[2], kTagPlane);
            outer(A0, B0, rho2 - el[1], A0, B0, rho2 - eh[1]);
            if (el[3] != 0.f) inner(A0, B0, rho2 - el[0], eh[3] != 0.f, A0, B0, rho2 - eh[0]);
        } else {
            // inside test on the same rounded constants as the roots, so that a
            // point counted inside never sees a root behind it
            auto cone = [&](const float* e, int a, float& A, float& B, float& C) {
                const float r0 = fmaf(e[a + 1], x[2], e[a]), rs = e[a + 1] * u[2];
                A = fmaf(-rs, rs, A0);
                B = fmaf(-r0, rs, B0);
                C = fmaf(-r0, r0, rho2);
            };
            float A, B, C, Ah, Bh, Ch;
            cone(el, 1, A, B, C);
            cone(eh, 1, Ah, Bh, Ch);
            m.in = fabsf(x[2]) <= el[0] && C <= 0.f;
            plane(2, el[0], eh[0], kTagPlane);
            outer(A, B, C, Ah, Bh, Ch);
            if (el[5] != 0.f) {
                cone(el, 3, A, B, C);
                cone(eh, 3, Ah, Bh, Ch);
                m.in = m.in && C >= 0.f;
                inner(A, B, C, eh[5] != 0.f, Ah, Bh, Ch);
            }
            if (ENTERED) crosses = false;   // (the double cone's other nappe: not argued)
        }
    }
    if (ENTERED) m.in = m.in || (entered && crosses && v.m64.kind < KTUBS);
    m.lo = fmaxf(m.lo, 0.f);
    m.hi = fmaxf(m.hi, 0.f);
    const float dt = 4.f * v.m32u.delta * r.inv_dn;
    if (!(m.in && m.lo > dt && fmaf(thi, 1.f + 32.f * kEps32f, dt) < second * (1.f - 32.f * kEps32f))) m.tag = kTagNone;
    return m;
}

// The same for a track inside the mother that starts between her shrunk copy and
// her surface: as one that has just entered.  (Without bounds of the exit such a
// track has the mother evaluated in FP64 first and its list after that: 524288
// tracks that all start there took 353 us in a batch of the toy detector, 101 so.)
// Out of line: rare among points anywhere in the mother.
static __device__ __noinline__ MotherExit mother_exit_near32(const VolView& v, Ray32 r) {
    return mother_exit32<true>(v, r, true);
}

// Which daughters the FP32 pass bounds: every daughter (filter_daughters),
// the uniform grid's walk (over the CSR lists, or over their staged short
// form), either one by the volume, or the daughters j_first, j_first + j_step,
// ... of the volume's own order (a share of them).
enum : int { kTravAll = 0, kTravGrid = 1, kTravEither = 2, kTravShare = 3, kTravGridSmall = 4 };

// the grid's lists in global memory
__device__ __forceinline__ GridTab grid_lists(const VolView& v) { return {nullptr, nullptr, v.vox_off, v.vox_fids, v.fhvy}; }

// FP32 pass: bounds of the mother and of the daughters.  When status == 1 on
// return, best/h already hold the final answer.  The FP64 track is taken from
// `src` (src(k): x, y, z, dx, dy, dz) where the rare FP64 paths need it again, so
// that a caller that holds it in shared memory need not keep it in registers.
template <int TRAV, bool SEGS = true, class Src>
__device__ __forceinline__ void refine_pass1(const VolView& v, const FiltTab& f, const GridTab& grid,
                                             const ShapeRec64* __restrict__ tab64, double px, double py, double pz,
                                             double qx, double qy, double qz, Src src, RefineState& st, double& best,
                                             int& h, int& nev, int j_first = 0, int j_step = 1) {
    nev = 0;
    st.status = 1;
    cands_clear(st.c);
    st.Lm = 0.f;
    if (!valid_track(px, py, pz, qx, qy, qz)) {
        best = d_nan();
        h = -2;
        return;
    }
    Ray32 r;
    r.p[0] = f64_to_f32_trunc(px); r.p[1] = f64_to_f32_trunc(py); r.p[2] = f64_to_f32_trunc(pz);
    r.d[0] = f64_to_f32_trunc(qx); r.d[1] = f64_to_f32_trunc(qy); r.d[2] = f64_to_f32_trunc(qz);
    const float dd = fmaf(r.d[0], r.d[0], fmaf(r.d[1], r.d[1], r.d[2] * r.d[2]));
    if (!(dd > v.dd_min && dd < 1e30f)) {
        // direction magnitude outside the range the FP32 bounds assume
        const double p[3] = {src(0), src(1), src(2)};
        if (contains64<SEGS>(v.m64, p))
            nav_all64_cold<SEGS>(v.m64, tab64, v.nd, p[0], p[1], p[2], src(3), src(4), src(5), best, h);
        else { best = 0.0; h = -2; }
        nev = 1000;
        return;
    }
    const float inv_dd = __frcp_rn(dd);
    r.inv_dn = rsqrtf(dd) * (1.f + 4.f * kEps32f);
#pragma unroll
    for (int k = 0; k < 3; ++k) r.e[k] = -r.d[k] * inv_dd;
    MotherExit m = mother_exit32(v, r);
    if (!m.in) {
        if (!contains64_cold<SEGS>(v.m64, src(0), src(1), src(2))) {
            best = 0.0;
            h = -2;
            return;
        }
        m = mother_exit_near32(v, r);
    }
    st.Lm = m.in ? fmaxf(lower_bound(m.lo, v.m32.delta, r.inv_dn), 0.f) : 0.f;
    const float Um = m.hi + 16.f * kEps32f * m.hi + v.m32u.delta * r.inv_dn;
    if (TRAV == kTravShare) {
        for (int j = j_first; j < v.nd; j += j_step) bound_daughter(v.d32[j], j, r, Um, st.c);
        cands_count(st.c);
    } else if (TRAV == kTravGridSmall) {
        filter_grid<true>(v, grid, r, Um, st.c);
    } else if (TRAV == kTravGrid || (TRAV == kTravEither && v.voxelized)) {
        filter_grid<false>(v, grid_lists(v), r, Um, st.c);
    } else {
        filter_daughters(f, r, Um, st.c);
    }
    st.tag = first_task(st) < 0 ? (v.m64.kind >= KTUBS ? kTagNone : m.tag) : st.c.j[0] >> kTagShift;
#pragma unroll
    for (int k = 0; k < kCand; ++k) st.c.j[k] &= kIdMask;
    st.status = 0;
}

// FP64 evaluation of one solid for one track (the mother's DistFromInside or
// a daughter's transform + DistFromOutside).
template <bool SEGS = true>
__device__ __forceinline__ double eval64(const VolView& v, const ShapeRec64* __restrict__ tab64, int j, double px,
                                         double py, double pz, double qx, double qy, double qz) {
    if (j < 0) {
        const double p[3] = {px, py, pz}, q[3] = {qx, qy, qz};
        return dist_in64<false, SEGS>(v.m64, p, q);
    }
    const ShapeRec64& r = tab64[j];
    double x[3], u[3];
    to_local64(r, px, py, pz, qx, qy, qz, x, u);
    return dist_out64<false, SEGS>(r, x, u);
}

// The FP64 step of solid r to the surface it is surely entered (a daughter) or
// left (the mother: `exit`) through: that surface's part of dist_out64 /
// dist_in64 with operations that round alike, so the same bits.  Planes and
// quadrics, tubes and cones run one code path with one division, so that the
// lanes of a warp need not be ordered by surface: an FP64 instruction costs a
// warp 64 cycles of its unit however few lanes take part, and a plane adds no
// instruction to a quadric's.
//  * A tube is a cone of slope 0 whose C = rho^2 - R^2 keeps the rounded R^2
//    (FMA(-1, R^2, rho^2); the other terms of slope 0 vanish exactly).
//  * The rising root of F = A s^2 + 2 B s + C is the falling root of -F (every
//    operation of a root commutes with the change of all signs).
//  * A plane needs one local coordinate; it is formed where a quadric forms its
//    first.
// ahead: (optional) the sign of the plane coordinate's direction.
__device__ __forceinline__ double surface64(const ShapeRec64& r, int tag, bool exit, double px, double py, double pz,
                                            double qx, double qy, double qz, bool* ahead = nullptr) {
    const double* d = r.d;
    const bool quad = tag == kTagOuter || tag == kTagInner, inner = tag == kTagInner;
    const int k = quad ? 0 : (tag >= kTagAxis ? tag - kTagAxis : 2);
    const double w0 = SUB(px, r.t[0]), w1 = SUB(py, r.t[1]), w2 = SUB(pz, r.t[2]);
    double xk, uk, x1 = w1, u1 = qy, x2 = w2, u2 = qz;
    if (r.flags & kRec64Identity) {
        xk = k == 0 ? w0 : (k == 1 ? w1 : w2);
        uk = k == 0 ? qx : (k == 1 ? qy : qz);
    } else {
        xk = FMA(r.R[6 + k], w2, FMA(r.R[3 + k], w1, MUL(r.R[k], w0)));
        uk = FMA(r.R[6 + k], qz, FMA(r.R[3 + k], qy, MUL(r.R[k], qx)));
        if (quad) {
            x1 = FMA(r.R[7], w2, FMA(r.R[4], w1, MUL(r.R[1], w0)));
            u1 = FMA(r.R[7], qz, FMA(r.R[4], qy, MUL(r.R[1], qx)));
            x2 = FMA(r.R[8], w2, FMA(r.R[5], w1, MUL(r.R[2], w0)));
            u2 = FMA(r.R[8], qz, FMA(r.R[5], qy, MUL(r.R[2], qx)));
        }
    }
    double num, den;
    bool ok = true;
    if (quad) {
        const bool tube = r.kind == KTUBE;
        const double b = tube ? 0.0 : (inner ? d[4] : d[2]);
        const double rho2 = DOT2(xk, xk, x1, x1);
        const double r0 = FMA(b, x2, tube ? 1.0 : (inner ? d[3] : d[1])), rs = MUL(b, u2);
        double A = FMA(-rs, rs, DOT2(uk, uk, u1, u1)), B = FMA(-r0, rs, DOT2(xk, uk, x1, u1));
        double C = FMA(-r0, tube ? (inner ? d[3] : d[4]) : r0, rho2);
        if (inner != exit) {   // rising
            A = -A;
            B = -B;
            C = -C;
        }
        const double D = FMA(B, B, -MUL(A, C));   // root_falling(A, B, C)
        const bool real = NONNEG(D);
        const bool bneg = IS_NEG(B);
        const double t = ADD(SQRT(real ? D : 1.0), fabs(B));
        num = bneg ? C : -t;
        den = bneg ? t : A;
        ok = real && (bneg || IS_NEG(A));
    } else {   // the face of axis k ahead (exit) or met first (entry)
        const double h = r.kind == KBOX ? d[k] : (r.kind == KTUBE ? d[2] : d[0]);
        const double c = copysign(h, uk);
        num = SUB(exit ? c : -c, xk);
        den = uk;
        if (ahead) *ahead = IS_POS(uk);
    }
    // one division for both kinds of lane (the empty statement keeps the
    // compiler from moving a copy of it into each branch)
    asm volatile("" : "+d"(num), "+d"(den));
    const double s = DIV(ok ? num : 1.0, ok ? den : 1.0);
    return ok ? s : d_inf();
}

// The answer of refine_rest() when no further FP64 evaluation can change it
// (nearly every track): the first task's value s_first is finite and every
// other bound -- the remaining candidates, the mother's when it was not the
// first task, the least evicted one -- lies above its FP32 upper bound.  A
// solid's FP64 value is at least its bound, so none of them can win or tie.
// Returns false when refine_rest() has to run.
__device__ __forceinline__ bool refine_fast(const RefineState& st, double s_first, double& best, int& h) {
    const bool mother_first = first_task(st) < 0;
    if (!LT(s_first, d_inf())) return false;
    const float up = f64_to_f32_up(s_first);
    const int k0 = mother_first ? 0 : 1;
#pragma unroll
    for (int k = 0; k < kCand; ++k)
        if (k >= k0 && k < st.c.n && st.c.L[k] <= up) return false;
    if (!mother_first && st.Lm <= up) return false;
    if (st.c.dropped <= up) return false;
    best = s_first;
    h = mother_first ? -1 : st.c.j[0];
    return true;
}

// FP64 refinement in ascending bound order, given the value s_first of the
// first task (first_task()).  Ties resolve as in Fig. 1a: mother, then the
// lowest index.  The bounds are compared in FP32 against best_up >= best, so
// at least every solid that could tie or win is refined (a solid refined in
// excess cannot change the answer).
template <bool SEGS = true>
static __device__ __noinline__ void refine_rest(const VolView& v, const ShapeRec64* __restrict__ tab64,
                                         const RefineState& st, double s_first, double px, double py, double pz,
                                         double qx, double qy, double qz, double& best, int& h, int& nev) {
    best = d_inf();
    h = -1;
    nev = 1;
    bool mdone;
    int k0;
    if (first_task(st) < 0) {
        mdone = true;
        best = s_first;   // the mother always beats +inf
        k0 = 0;
    } else {
        mdone = false;
        if (LT(s_first, best)) {
            best = s_first;
            h = st.c.j[0];
        }
        k0 = 1;
    }
    float best_up = f64_to_f32_up(best);
#pragma unroll
    for (int k = 0; k < kCand; ++k) {
        if (k >= k0 && k < st.c.n) {
            const float L = st.c.L[k];
            if (!mdone && st.Lm <= L) {
                const double sm = eval64<SEGS>(v, tab64, -1, px, py, pz, qx, qy, qz);
                ++nev;
                mdone = true;
                if (LE(sm, best)) {
                    best = sm;
                    h = -1;
                    best_up = f64_to_f32_up(best);
                }
            }
            if (L <= best_up) {
                const int j = st.c.j[k];
                const double s = eval64<SEGS>(v, tab64, j, px, py, pz, qx, qy, qz);
                ++nev;
                // same order as the sequential loop: bit-pattern order of
                // non-negative steps, ties to the mother, then the lowest index
                if (LT(s, best) || (BITS(s) == BITS(best) && h >= 0 && j < h)) {
                    best = s;
                    h = j;
                    best_up = f64_to_f32_up(best);
                }
            }
        }
    }
    if (!mdone && st.Lm <= best_up) {
        const double sm = eval64<SEGS>(v, tab64, -1, px, py, pz, qx, qy, qz);
        ++nev;
        if (LE(sm, best)) {
            best = sm;
            h = -1;
            best_up = f64_to_f32_up(best);
        }
    }
    if (st.c.dropped <= best_up) {
        nav_all64_cold<SEGS>(v.m64, tab64, v.nd, px, py, pz, qx, qy, qz, best, h);
        nev += 1000;   // marks a fallback in the statistics
    }
}

// a track whose first task is not certain: the whole solid (rare, out of line; tubes
// and cones in one path, since a warp may hold both)
static __device__ __noinline__ double eval64_cold(const VolView& v, const ShapeRec64* __restrict__ tab64, int j, double px,
                                                  double py, double pz, double qx, double qy, double qz) {
    if (j < 0) return eval64<false>(v, tab64, j, px, py, pz, qx, qy, qz);
    const ShapeRec64& r = tab64[j];
    double x[3], u[3];
    to_local64(r, px, py, pz, qx, qy, qz, x, u);
    return r.kind == KBOX ? box_out64(r.d, x, u) : quad_out64(r, x, u);
}

// The FP64 part of a track after its FP32 pass.
__device__ __forceinline__ void finish_direct(const VolView& v, const ShapeRec64* __restrict__ tab64, const ShapeRec64& m64,
                                              const RefineState& rs, double px, double py, double pz, double qx,
                                              double qy, double qz, double& best, int& h, int& nev) {
    if (rs.status != 0) return;
    const int task = first_task(rs);
    double s1;
    if (rs.tag != kTagNone) s1 = surface64(task < 0 ? m64 : tab64[task], rs.tag, task < 0, px, py, pz, qx, qy, qz);
    else s1 = eval64_cold(v, tab64, task, px, py, pz, qx, qy, qz);
    nev = 1;
    if (!refine_fast(rs, s1, best, h)) refine_rest<false>(v, tab64, rs, s1, px, py, pz, qx, qy, qz, best, h, nev);
}

}  // namespace geonav
