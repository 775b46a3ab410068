// nav_common.cuh -- the FP64 navigator step of Fig. 1 for one track, shared by
// the plain FP64 kernel and by the fallback of the FP32-filter kernel, so
// both produce bit-identical answers.
#pragma once
#include "geo_internal.h"
#include "shapes64.cuh"

namespace geonav {

// Invalid input (non-finite or zero direction): NaN, -2.  Returns false.
// (exponent bits checked with integer operations)
__device__ __forceinline__ bool finite64(double a) { return (BITS(a) & kAbsMask) < 0x7ff0000000000000LL; }
__device__ __forceinline__ bool valid_track(double px, double py, double pz, double qx, double qy, double qz) {
    const bool finite = finite64(px) && finite64(py) && finite64(pz) && finite64(qx) && finite64(qy) &&
                        finite64(qz);
    return finite && !(IS_ZERO(qx) && IS_ZERO(qy) && IS_ZERO(qz));
}

// tube_out64 and cone_out64 (no apex on an end plane) in one path, so that
// lanes with either kind run it together: a tube is a cone of slope 0 whose
// outer and inner C keep the rounded squares of its radii (surface64 in
// nav_refine.cuh has the argument that the bits are the same).
__device__ __forceinline__ double quad_out64(const ShapeRec64& r, const double* x, const double* u) {
    const double* d = r.d;
    const bool tube = r.kind == KTUBE;
    const double dz = tube ? d[2] : d[0], bo = tube ? 0.0 : d[2], bi = tube ? 0.0 : d[4];
    const double rho2 = rho2_of(x);
    // -1 * R^2 (tube), -R * R (cone)
    const double ro0 = tube ? 1.0 : FMA(bo, x[2], d[1]), ri0 = tube ? 1.0 : FMA(bi, x[2], d[3]);
    const double ro1 = tube ? d[4] : ro0, ri1 = tube ? d[3] : ri0;
    const bool hole = tube ? IS_POS(d[0]) : !IS_ZERO(d[11]);
    if (ABS_LE(x[2], dz) && LE(rho2, MUL(ro0, ro1)) && (!hole || LE(MUL(ri0, ri1), rho2))) return 0.0;
    double best = d_inf();
    const bool zc = ABS_GT(x[2], dz) && OPPOSITE(x[2], u[2]);
    if (zc) {   // the z-plane the track approaches from outside the slab
        const double t = DIV(SUB(copysign(dz, x[2]), x[2]), u[2]);
        const double xh = FMA(t, u[0], x[0]), yh = FMA(t, u[1], x[1]);
        const double r2 = DOT2(xh, xh, yh, yh);
        const double lo2 = tube ? d[3] : (IS_POS(x[2]) ? d[7] : d[5]);
        const double hi2 = tube ? d[4] : (IS_POS(x[2]) ? d[8] : d[6]);
        if (LE(r2, hi2) && LE(lo2, r2)) best = t;
    }
    const double A0 = DOT2(u[0], u[0], u[1], u[1]);
    const double B0 = DOT2(x[0], u[0], x[1], u[1]);
    {   // outer surface, crossed inwards
        const double rs = MUL(bo, u[2]);
        const double s = root_falling(FMA(-rs, rs, A0), FMA(-ro0, rs, B0), FMA(-ro0, ro1, rho2));
        if (NONNEG(s) && LT(s, best) && ABS_LE(FMA(s, u[2], x[2]), dz)) best = s;
    }
    if (hole) {   // inner surface, crossed outwards (out of the hole)
        const double rs = MUL(bi, u[2]);
        const double s = root_rising(FMA(-rs, rs, A0), FMA(-ri0, rs, B0), FMA(-ri0, ri1, rho2));
        if (NONNEG(s) && LT(s, best) && ABS_LE(FMA(s, u[2], x[2]), dz)) best = s;
    }
    return best;
}

// Mother DistFromInside, then for every daughter: bounding-sphere test against
// the current best, master->local transform, DistFromOutside, strict '<'
// (mother first, then the lowest index win ties).  Track assumed valid and
// inside the mother.
template <bool SEGS = true>
__device__ __forceinline__ void nav_all64(const ShapeRec64& m, const ShapeRec64* __restrict__ tab, int nd,
                                          double px, double py, double pz, double qx, double qy, double qz,
                                          double& best, int& h) {
    const double p[3] = {px, py, pz}, q[3] = {qx, qy, qz};
    best = dist_in64<false, SEGS>(m, p, q);
    h = -1;
    const double dd = qx * qx + qy * qy + qz * qz;
    const double dn = sqrt(dd);
    for (int j = 0; j < nd; ++j) {
        const ShapeRec64& r = tab[j];
        // bounding sphere about t: centre parameter proj/dd, radius brad/|d|
        // (brad is enlarged on the host, so these culls are conservative)
        const double w0 = r.t[0] - px, w1 = r.t[1] - py, w2 = r.t[2] - pz;
        const double proj = w0 * qx + w1 * qy + w2 * qz;
        const double rb = r.brad * dn;
        if (proj + rb < 0.0) continue;                  // sphere entirely behind
        if (proj - rb >= best * dd) continue;           // sphere starts beyond best
        const double ww = w0 * w0 + w1 * w1 + w2 * w2;
        if (ww * dd - proj * proj > rb * rb) continue;  // line misses the sphere
        double x[3], u[3];
        to_local64(r, px, py, pz, qx, qy, qz, x, u);
        const double s = dist_out64<false, SEGS>(r, x, u);
        if (LT(s, best)) {
            best = s;
            h = j;
        }
    }
}

// The same step with the uniform grid: cells are walked in ray order (FP64
// 3D-DDA) and the walk stops once the best step lies before the exit of the
// cell just finished (with a relative margin of 2^-40): every daughter the
// track could still enter starts in a later cell.  Daughters arrive out of
// index order, so ties are resolved explicitly (mother, then lowest index).
__device__ __forceinline__ void nav_vox64(const VolView& v, const ShapeRec64* __restrict__ tab, double px,
                                          double py, double pz, double qx, double qy, double qz, double& best,
                                          int& h) {
    const double p[3] = {px, py, pz}, q[3] = {qx, qy, qz};
    best = dist_in64(v.m64, p, q);
    h = -1;
    const double dd = qx * qx + qy * qy + qz * qz;
    const double dn = sqrt(dd);
    int i0, i1, i2, s0, s1, s2;
    double m0, m1, m2, e0, e1, e2;
    auto setup = [&](int k, int& ii, int& st, double& tm, double& te) {
        const int g = v.grid[k];
        ii = int(floor((p[k] - v.lo[k]) * v.inv_cell[k]));
        ii = ii < 0 ? 0 : (ii >= g ? g - 1 : ii);
        if (q[k] > 0.0) {
            st = 1;
            tm = (v.lo[k] + (ii + 1) * v.cell[k] - p[k]) / q[k];
            te = v.cell[k] / q[k];
        } else if (q[k] < 0.0) {
            st = -1;
            tm = (v.lo[k] + ii * v.cell[k] - p[k]) / q[k];
            te = -v.cell[k] / q[k];
        } else {
            st = 0;
            tm = d_inf();
            te = d_inf();
        }
    };
    setup(0, i0, s0, m0, e0);
    setup(1, i1, s1, m1, e1);
    setup(2, i2, s2, m2, e2);
    const int g0 = v.grid[0], g1 = v.grid[1], g2 = v.grid[2];
    int mb0 = -1, mb1 = -1, mb2 = -1, mb3 = -1;
    int left = g0 + g1 + g2 + 3;   // cells at most
    int c = (i0 * g1 + i1) * g2 + i2, e = v.vox_off[c], q1 = v.vox_off[c + 1];
    // A flat walk: every lane goes on by itself, a list entry or a cell a turn, until it
    // holds a daughter whose sphere it meets, and all lanes evaluate theirs together.
    // (As two nested loops the lanes' evaluations were together or apart as the
    // compiler happened to place them: 512 daughters, 2^20 tracks, 3.6 to 5.3 ms
    // for 2.94 so.)
    bool more = true;
    while (more) {
        int j = -1;
        do {
            if (e < q1) {
                const int k = v.vox_ids[e++];
                if (k != mb0 && k != mb1 && k != mb2 && k != mb3) {
                    mb3 = mb2; mb2 = mb1; mb1 = mb0; mb0 = k;
                    const ShapeRec64& r = tab[k];
                    const double w0 = r.t[0] - px, w1 = r.t[1] - py, w2 = r.t[2] - pz;
                    const double proj = w0 * qx + w1 * qy + w2 * qz;
                    const double rb = r.brad * dn;
                    const double ww = w0 * w0 + w1 * w1 + w2 * w2;
                    if (!(proj + rb < 0.0) && !(proj - rb > best * dd) && !(ww * dd - proj * proj > rb * rb)) j = k;
                }
            } else {
                // the cell is left at min(m0, m1, m2): nothing entered later can win
                const double mn = fmin(m0, fmin(m1, m2));
                const bool a0 = m0 <= m1 && m0 <= m2, a1 = !a0 && m1 <= m2, a2 = !a0 && !a1;
                i0 += a0 ? s0 : 0;
                i1 += a1 ? s1 : 0;
                i2 += a2 ? s2 : 0;
                m0 = a0 ? m0 + e0 : m0;
                m1 = a1 ? m1 + e1 : m1;
                m2 = a2 ? m2 + e2 : m2;
                more = !(best < mn * (1.0 - 9.094947017729282e-13)) && i0 >= 0 && i0 < g0 && i1 >= 0 && i1 < g1 && i2 >= 0 &&
                       i2 < g2 && --left > 0;
                if (more) {
                    c = (i0 * g1 + i1) * g2 + i2;
                    e = v.vox_off[c];
                    q1 = v.vox_off[c + 1];
                }
            }
        } while (j < 0 && more);
        if (j >= 0) {
            double x[3], u[3];
            to_local64(tab[j], px, py, pz, qx, qy, qz, x, u);
            const double s = dist_out64(tab[j], x, u);
            if (LT(s, best) || (BITS(s) == BITS(best) && h >= 0 && j < h)) {
                best = s;
                h = j;
            }
        }
    }
}

__device__ __forceinline__ void store_result(int64_t i, int64_t n, double best, int h, double px, double py,
                                             double pz, double qx, double qy, double qz, double* step,
                                             int32_t* hit, double* bpoint) {
    step[i] = best;
    hit[i] = h;
    if (bpoint) {
        bpoint[i] = FMA(best, qx, px);
        bpoint[n + i] = FMA(best, qy, py);
        bpoint[2 * n + i] = FMA(best, qz, pz);
    }
}

}  // namespace geonav
