// nav_fp64.cu -- the plain FP64 vector navigator of Fig. 1b on the GPU (and,
// for small baskets, its warp-per-track form with a shuffle (step, index)
// minimum), and the navigator-level Contains and Safety of Sec. 3.1.
//
// One thread per track (grid-stride over the basket).  The basket is read as
// coalesced FP64 structure-of-arrays.  Mother first, then the daughters that a
// cull in FP64 does not exclude, a running (step, index) minimum (mother, then the
// lowest index win ties).
#include <cuda_runtime.h>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "shapes64.cuh"
#include "stage.cuh"

namespace geonav {

// Voxelised volumes: the grid's walk (nav_vox64), bound by the FP64 unit (its walk's
// and culls' instructions).  512 daughters: 65536 tracks 290 -> 241 us, 2^20 3.64 -> 2.94 ms;
// the records staged in shared memory give the same times (2.95 ms).
__global__ void __launch_bounds__(256) k_dist_vox64(VolView v, Basket b, double* __restrict__ step,
                                                    int32_t* __restrict__ hit, double* __restrict__ bpoint) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
        double best;
        int h;
        const double p[3] = {px, py, pz};
        if (!valid_track(px, py, pz, qx, qy, qz)) {
            best = d_nan();
            h = -2;
        } else if (!contains64(v.m64, p)) {
            best = 0.0;
            h = -2;
        } else {
            nav_vox64(v, v.d64, px, py, pz, qx, qy, qz, best, h);
        }
        store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
    }
}

template <bool SEGS>
static __device__ __noinline__ void nav_all64_far(const ShapeRec64& m, const ShapeRec64* __restrict__ tab, int nd,
                                                  double px, double py, double pz, double qx, double qy, double qz,
                                                  double& best, int& h) {
    nav_all64<SEGS>(m, tab, nd, px, py, pz, qx, qy, qz, best, h);
}

// Every daughter, all in FP64, in the filter's order (filter_pass.cuh has the
// scheme and its reasons): culls for all lanes together -- bounding spheres,
// and bounding annuli of unrotated tubes and cones -- then each lane its own
// daughters, of the annuli the two that start nearest first.  The culls
// compare on bit patterns, so an annulus costs 8 FP64 instructions and a
// sphere 12.  `tab`: the FP64 records.
template <bool SEGS>
__device__ __forceinline__ void nav_lists64(const VolView& v, const Cull64* __restrict__ C,
                                            const ShapeRec64* __restrict__ tab, double px, double py, double pz,
                                            double qx, double qy, double qz, double& best, int& h) {
    const double p[3] = {px, py, pz}, q[3] = {qx, qy, qz};
    best = dist_in64<false, SEGS>(v.m64, p, q);
    h = -1;
    const double perp2 = DOT2(qx, qx, qy, qy), dd = FMA(qz, qz, perp2), dn = SQRT(dd);
    if (!(LT(1e-200, dd) && LT(dd, 1e200))) {   // the culls' squares could leave the range of a double
        nav_all64_far<SEGS>(v.m64, v.d64, v.nd, px, py, pz, qx, qy, qz, best, h);
        return;
    }
    double inv_z = 0.0, inv_r = 0.0;
    if (v.nq1 > 0) {
        // lowered below any rounding of the products; no radial bound along the axis
        constexpr double kLow = 1.0 - 0x1p-48;
        inv_z = MUL(DIV(1.0, fabs(qz)), kLow);
        inv_r = LT(MUL(dd, 1e-24), perp2) ? MUL(DIV(1.0, SQRT(perp2)), kLow) : 0.0;
    }
    auto eval = [&](int j) {
        const ShapeRec64& r = tab[j];
        double x[3], u[3];
        to_local64(r, px, py, pz, qx, qy, qz, x, u);
        double s;
        if (!SEGS && r.kind != KBOX) s = quad_out64(r, x, u);
        else s = dist_out64<false, SEGS>(r, x, u);
        if (LT(s, best) || (BITS(s) == BITS(best) && h >= 0 && j < h)) {
            best = s;
            h = j;
        }
    };
    double rho = 0.0, rr = 0.0;   // distance to the axis: the start's, the forward ray's least
    auto to_axis = [&](const Cull64& c) {
        const double wx = SUB(px, c.t[0]), wy = SUB(py, c.t[1]);
        rho = SQRT(DOT2(wx, wx, wy, wy));
        const double away = DOT2(wx, qx, wy, qy);
        rr = NONNEG(away) ? rho : MUL(fabs(FMA(wx, qy, -MUL(wy, qx))), inv_r);
    };
    auto pos = [](double a) { return BITS(a) < 0 ? 0.0 : a; };   // max(a, 0)
    // start of the annulus' part of the track, +inf when it is missed or starts beyond best
    auto annulus = [&](const Cull64& c) {
        const double wz = SUB(pz, c.t[2]), wzs = BITS(qz) < 0 ? -wz : wz;
        const double t_in = pos(MUL(SUB(-c.h, wzs), inv_z)), t_out = MUL(SUB(c.h, wzs), inv_z);
        const double t_r = MUL(MAXP(pos(SUB(rho, c.a)), pos(SUB(c.b, rho))), inv_r);
        const double L = MAXP(t_in, t_r);
        // (t_out is lowered like L: compared with a margin of its own)
        const bool miss = BITS(t_out) < 0 || BITS(t_out) + (1LL << 8) < BITS(L) || LT(c.a, rr) || LT(best, L);
        return miss ? d_inf() : L;
    };
    for (int base = 0; base < v.nf; base += 32) {
        const Cull64* S = C + base;
        const int cnt = min(32, v.nf - base), n1 = max(0, min(cnt, v.nq1 - base));
        unsigned m = 0;
        double l1 = d_inf(), l2 = d_inf();
        int k1 = -1, k2 = -1, k = 0;
        for (; k < n1; ++k) {
            if (S[k].axis) to_axis(S[k]);   // warp-uniform: another axis than the solid before
            const double L = annulus(S[k]);
            if (!LT(L, d_inf())) continue;
            m |= 1u << k;
            if (LT(L, l1)) {
                l2 = l1;
                k2 = k1;
                l1 = L;
                k1 = k;
            } else if (LT(L, l2)) {
                l2 = L;
                k2 = k;
            }
        }
        for (; k < cnt; ++k) {
            const double w0 = SUB(S[k].t[0], px), w1 = SUB(S[k].t[1], py), w2 = SUB(S[k].t[2], pz);
            const double proj = FMA(w2, qz, FMA(w1, qy, MUL(w0, qx)));
            const double ww = FMA(w2, w2, FMA(w1, w1, MUL(w0, w0)));
            // squared distance of the line times dd against the radius' (a filling entry's is negative)
            const double far2 = FMA(-proj, proj, MUL(ww, dd)), rb2 = MUL(S[k].a, dd);
            if (BITS(rb2) < 0 || LT(rb2, pos(far2))) continue;
            const double rb = MUL(S[k].b, dn);
            if (BITS(ADD(proj, rb)) < 0 || LT(MUL(best, dd), pos(SUB(proj, rb)))) continue;   // behind, beyond
            m |= 1u << k;
        }
        if (k1 >= 0) m &= ~(1u << k1);
        if (k2 >= 0) m &= ~(1u << k2);
        for (;;) {
            int w = k1;
            k1 = k2;
            k2 = -1;
            if (w >= 0 && LT(best, l1)) w = -1;
            l1 = l2;
            if (w < 0) {
                if (k1 >= 0) continue;
                if (!m) break;
                w = __ffs(m) - 1;
                m &= m - 1;
                if (w < n1) {
                    to_axis(S[w]);
                    if (!LT(annulus(S[w]), d_inf())) continue;
                }
            }
            eval(S[w].id);
        }
    }
}

// What bounds it: the FP64 unit (66 %; 1050 FP64 warp instructions per 32 tracks
// of the toy detector, 2200 when the warp walked the daughters together).
// 100003 tracks: 484 -> 242 us.  Blocks of 64 threads, eight per SM: the last
// wave's imbalance costs least (128 x 5 259 us, 128 x 8 258, 32 x 20 238).
constexpr int kFp64Threads = 64, kFp64Blocks = 8;
constexpr int kFp64Tables = 24 * 1024;   // bytes staged per block

// STAGED: 1 the cull table, 2 the FP64 records too
template <int STAGED, bool SEGS>
__global__ void __launch_bounds__(kFp64Threads, kFp64Blocks)
    k_dist_fp64(const __grid_constant__ VolView v, Basket b, double* __restrict__ step, int32_t* __restrict__ hit,
                double* __restrict__ bpoint) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    const Cull64* C = v.cull;
    const ShapeRec64* tab = v.d64;
    if (STAGED) {
        const uint32_t bc = uint32_t(v.nf) * uint32_t(sizeof(Cull64));
        if (!stage_tables(smem_raw, v.cull, bc, smem_raw + bc, v.d64,
                          STAGED == 2 ? uint32_t(v.nd) * uint32_t(sizeof(ShapeRec64)) : 0, &bar, v.status))
            return;
        C = reinterpret_cast<const Cull64*>(smem_raw);
        if (STAGED == 2) tab = reinterpret_cast<const ShapeRec64*>(smem_raw + bc);
    }
    const int64_t stride = int64_t(gridDim.x) * kFp64Threads;
    for (int64_t i = int64_t(blockIdx.x) * kFp64Threads + threadIdx.x; i < b.n; i += stride) {
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
        double best;
        int h;
        const double p[3] = {px, py, pz};
        if (!valid_track(px, py, pz, qx, qy, qz)) {
            best = d_nan();
            h = -2;
        } else if (!contains64<SEGS>(v.m64, p)) {
            best = 0.0;
            h = -2;
        } else {
            nav_lists64<SEGS>(v, C, tab, px, py, pz, qx, qy, qz, best, h);
        }
        store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
    }
}

// Small baskets: one warp per track.  The lanes take the daughters j = lane,
// lane + 32, ... (bounding-sphere cull against the mother's step), each keeps
// its (step, index) minimum with strict '<', and the warp reduces the pairs
// with shuffles (smaller step, then smaller index); the mother (index -1)
// wins ties.  That is the thread-per-track loop's answer bit for bit: it
// takes the daughters in index order with strict '<' after the mother, and
// a daughter it culls against its running best could not have won (the cull
// is conservative), so the lanes' weaker culls only evaluate more.  Every
// lane computes the track's mother step and containment (warp-uniform: the
// FP64 pipe charges a warp instruction whatever the active lanes).  The
// table is read through L1: a few tracks would not repay its staging.
template <bool SEGS>
__global__ void __launch_bounds__(256) k_dist_warp(VolView v, Basket b, double* __restrict__ step,
                                                   int32_t* __restrict__ hit, double* __restrict__ bpoint) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < b.n; i += nwarps) {
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
        const double p[3] = {px, py, pz}, q[3] = {qx, qy, qz};
        double best;
        int h;
        if (!valid_track(px, py, pz, qx, qy, qz)) {
            best = d_nan();
            h = -2;
        } else if (!contains64<SEGS>(v.m64, p)) {
            best = 0.0;
            h = -2;
        } else {
            const double sm = dist_in64<false, SEGS>(v.m64, p, q);
            const double dd = qx * qx + qy * qy + qz * qz;
            const double dn = sqrt(dd);
            double lb = d_inf();
            int lh = 0x7fffffff;
            for (int j = lane; j < v.nd; j += 32) {
                const ShapeRec64& r = v.d64[j];
                const double w0 = r.t[0] - px, w1 = r.t[1] - py, w2 = r.t[2] - pz;
                const double proj = w0 * qx + w1 * qy + w2 * qz;
                const double rb = r.brad * dn;
                if (proj + rb < 0.0) continue;
                if (proj - rb >= sm * dd) continue;
                const double ww = w0 * w0 + w1 * w1 + w2 * w2;
                if (ww * dd - proj * proj > rb * rb) continue;
                double x[3], u[3];
                to_local64(r, px, py, pz, qx, qy, qz, x, u);
                const double sj = dist_out64<false, SEGS>(r, x, u);
                if (LT(sj, lb)) {
                    lb = sj;
                    lh = j;
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, lb, off);
                const int oh = __shfl_xor_sync(0xffffffffu, lh, off);
                if (LT(ob, lb) || (BITS(ob) == BITS(lb) && oh < lh)) {
                    lb = ob;
                    lh = oh;
                }
            }
            best = sm;
            h = -1;
            if (LT(lb, sm)) {
                best = lb;
                h = lh;
            }
        }
        if (lane == 0) store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
    }
}

template <bool SMEM>
__global__ void __launch_bounds__(256) k_contains(VolView v, Basket b, int32_t* __restrict__ where) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    const ShapeRec64* tab = v.d64;
    if (SMEM) {
        if (!stage_table(smem_raw, v.d64, uint32_t(v.nd) * sizeof(ShapeRec64), &bar, v.status)) return;
        tab = reinterpret_cast<const ShapeRec64*>(smem_raw);
    }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const double p[3] = {b.x[i], b.y[i], b.z[i]};
        int w = -2;
        if (contains64(v.m64, p)) {
            w = -1;
            for (int j = 0; j < v.nd; ++j) {
                const ShapeRec64& r = tab[j];
                const double w0 = p[0] - r.t[0], w1 = p[1] - r.t[1], w2 = p[2] - r.t[2];
                if (w0 * w0 + w1 * w1 + w2 * w2 > r.brad * r.brad) continue;
                double x[3], u[3];
                to_local64(r, p[0], p[1], p[2], 0.0, 0.0, 0.0, x, u);
                if (contains64(r, x)) {
                    w = j;
                    break;
                }
            }
        }
        where[i] = w;
    }
}

template <bool SMEM>
__global__ void __launch_bounds__(256) k_safety_fp64(VolView v, Basket b, double* __restrict__ saf) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    const ShapeRec64* tab = v.d64;
    if (SMEM) {
        if (!stage_table(smem_raw, v.d64, uint32_t(v.nd) * sizeof(ShapeRec64), &bar, v.status)) return;
        tab = reinterpret_cast<const ShapeRec64*>(smem_raw);
    }
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const double p[3] = {b.x[i], b.y[i], b.z[i]};
        double s = 0.0;
        if (contains64(v.m64, p)) {
            s = safety64(v.m64, p, true);
            for (int j = 0; j < v.nd && s > 0.0; ++j) {
                const ShapeRec64& r = tab[j];
                const double w0 = p[0] - r.t[0], w1 = p[1] - r.t[1], w2 = p[2] - r.t[2];
                const double c = sqrt(w0 * w0 + w1 * w1 + w2 * w2);
                if (c - r.brad >= s) continue;   // the whole daughter is farther than s
                double x[3], u[3];
                to_local64(r, p[0], p[1], p[2], 0.0, 0.0, 0.0, x, u);
                s = fmin(s, safety64(r, x, false));
            }
        }
        saf[i] = s;
    }
}

// ------------------------------------------------------------ launchers ---

#define GEO_LAUNCH(KER, ...)                                                                 \
    do {                                                                                     \
        const int smem = v.smem64 ? v.nd * int(sizeof(ShapeRec64)) : 0;                      \
        if (v.smem64) {                                                                      \
            cudaError_t e = prep(KER<true>, smem);                                           \
            if (e != cudaSuccess) return e;                                                  \
            KER<true><<<blocks_for(KER<true>, b.n, smem, num_sms), 256, smem, s>>>(__VA_ARGS__); \
        } else {                                                                             \
            KER<false><<<blocks_for(KER<false>, b.n, 0, num_sms), 256, 0, s>>>(__VA_ARGS__);   \
        }                                                                                    \
        return cudaGetLastError();                                                           \
    } while (0)

// One warp per track, in both modes, when the basket is small (at most 8 tracks per
// SM: the latency of a track's serial daughter loop would set the time) and the
// daughters fit one pass of the lanes (at most 32).  With more daughters, or
// more tracks, the warp's FP64 instructions -- charged in full whatever the
// lanes that take part -- outweigh the latency it hides.  Per call (graphs of 20
// calls), the kernel that would take the basket otherwise -> this one, 16 and 1024 tracks:
// GEO_FP64 (lists per lane) four boxes 8.3 -> 8.1 and 10.5 -> 8.6 us, eight solids of
// the toy detector 13.7 -> 15.6 and 17.7 -> 18.2, four polycones 21.2 -> 15.3 and 61.4
// -> 22.7; GEO_FP32_REFINE four polycones (pipelined) 14.8 -> 15.5 and 48.7 -> 22.7.
// (The direct kernel, newer than this rule, would take 4.2 and 5.1 us for the boxes and
// 6.3 and 11.7 for the eight solids.)
bool small_basket(const VolView& v, int64_t n, int num_sms) {
    return !v.voxelized && v.nd <= 32 && n <= int64_t(8) * num_sms;
}

cudaError_t launch_dist_warp(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                             cudaStream_t s, int num_sms) {
    if (v.segs) {
        k_dist_warp<true><<<blocks_for(k_dist_warp<true>, b.n * 32, 0, num_sms), 256, 0, s>>>(v, b, step, hit,
                                                                                             bpoint);
    } else {
        k_dist_warp<false><<<blocks_for(k_dist_warp<false>, b.n * 32, 0, num_sms), 256, 0, s>>>(v, b, step, hit,
                                                                                               bpoint);
    }
    return cudaGetLastError();
}

template <int STAGED, bool SEGS>
static cudaError_t launch_fp64(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint, int smem,
                               cudaStream_t s, int num_sms) {
    cudaError_t e = prep(k_dist_fp64<STAGED, SEGS>, smem);
    if (e != cudaSuccess) return e;
    k_dist_fp64<STAGED, SEGS><<<blocks_for(k_dist_fp64<STAGED, SEGS>, b.n, smem, num_sms, kFp64Threads), kFp64Threads, smem,
                                s>>>(v, b, step, hit, bpoint);
    return cudaGetLastError();
}

cudaError_t launch_dist_fp64(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                             cudaStream_t s, int num_sms) {
    if (small_basket(v, b.n, num_sms)) return launch_dist_warp(v, b, step, hit, bpoint, s, num_sms);
    if (v.voxelized) {
        k_dist_vox64<<<blocks_for(k_dist_vox64, b.n, 0, num_sms), 256, 0, s>>>(v, b, step, hit, bpoint);
        return cudaGetLastError();
    }
    const int64_t bc = int64_t(v.nf) * int64_t(sizeof(Cull64)), br = bc + int64_t(v.nd) * int64_t(sizeof(ShapeRec64));
    const int staged = br <= kFp64Tables ? 2 : (bc <= kFp64Tables ? 1 : 0);
    const int smem = staged == 2 ? int(br) : (staged == 1 ? int(bc) : 0);
    switch (2 * staged + (v.segs ? 1 : 0)) {
        case 0: return launch_fp64<0, false>(v, b, step, hit, bpoint, smem, s, num_sms);
        case 1: return launch_fp64<0, true>(v, b, step, hit, bpoint, smem, s, num_sms);
        case 2: return launch_fp64<1, false>(v, b, step, hit, bpoint, smem, s, num_sms);
        case 3: return launch_fp64<1, true>(v, b, step, hit, bpoint, smem, s, num_sms);
        case 4: return launch_fp64<2, false>(v, b, step, hit, bpoint, smem, s, num_sms);
        default: return launch_fp64<2, true>(v, b, step, hit, bpoint, smem, s, num_sms);
    }
}

cudaError_t launch_contains(const VolView& v, const Basket& b, int32_t* where, int mode, cudaStream_t s,
                            int num_sms) {
    if (mode == GEO_FP32_REFINE) return launch_contains_filter(v, b, where, s, num_sms);
    GEO_LAUNCH(k_contains, v, b, where);
}

cudaError_t launch_safety(const VolView& v, const Basket& b, double* saf, int mode, cudaStream_t s,
                          int num_sms) {
    if (mode == GEO_FP32_REFINE) return launch_safety_filter(v, b, saf, s, num_sms);
    if (mode == GEO_SAFETY_ESTIMATE) return launch_safety_estimate(v, b, saf, s, num_sms);
    GEO_LAUNCH(k_safety_fp64, v, b, saf);
}

}  // namespace geonav
