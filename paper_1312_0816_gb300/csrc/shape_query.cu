// shape_query.cu -- the elementary per-shape algorithms of Sec. 3.1 on their
// own (the vectorised DistFromOutside / DistFromInside / Safety / Contains of
// one solid that Fig. 2 measures per shape), for a basket of points or tracks.
//
// The solid's FP64 record travels in the kernel parameters (every lane reads
// the same constants), and so does a polycone's plane table (read through
// the address of the __grid_constant__ parameter, so the call allocates
// nothing); each thread takes one track, applies the placement's
// master->local transform and the FP64 routine of the navigator kernels
// (shapes64.cuh), so the values are the ones the navigator computes for that
// solid.  Grid-stride over the basket, blocks sized by occupancy.
#include <cuda_runtime.h>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "nav_refine.cuh"
#include "point_pass.cuh"
#include "shapes64.cuh"

namespace geonav {

template <int WHAT>
__global__ void __launch_bounds__(256) k_shape(const __grid_constant__ ShapeArg a, Basket b, double* __restrict__ out,
                                               int32_t* __restrict__ face) {
    const ShapeRec64& r = a.r;
    const bool pc = r.kind == KPCON;
    const double* T = a.table;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        double v;
        int f = -1;
        if (WHAT == GEO_Q_DIST_OUT || WHAT == GEO_Q_DIST_IN) {
            const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
            if (!valid_track(px, py, pz, qx, qy, qz)) {
                v = d_nan();
            } else {
                double x[3], u[3];
                to_local64(r, px, py, pz, qx, qy, qz, x, u);
                if (WHAT == GEO_Q_DIST_OUT) {
                    v = pc ? pcon_out64_call<true, false>(r.d, T, x[0], x[1], x[2], u[0], u[1], u[2], &f)
                           : dist_out64<true>(r, x, u, &f);
                } else if (pc ? pcon_contains64(r.d, T, x[0], x[1], x[2]) : contains64(r, x)) {
                    v = pc ? pcon_in64_call<true>(r.d, T, x[0], x[1], x[2], u[0], u[1], u[2], &f)
                           : dist_in64<true>(r, x, u, &f);
                } else {
                    v = 0.0;   // DistFromInside of a point outside
                }
            }
        } else {
            const bool fin = finite64(px) && finite64(py) && finite64(pz);
            double x[3];
            point_to_local64(r, px, py, pz, x);
            const bool in = fin && (pc ? pcon_contains64(r.d, T, x[0], x[1], x[2]) : contains64(r, x));
            if (!fin) v = d_nan();
            else if (WHAT == GEO_Q_CONTAINS) v = in ? 1.0 : 0.0;
            else if (pc) v = in == (WHAT == GEO_Q_SAFETY_IN) ? pcon_safety64(r.d, T, x[0], x[1], x[2], in) : 0.0;
            else v = safety64(r, x, WHAT == GEO_Q_SAFETY_IN);
        }
        out[i] = v;
        if (face) face[i] = f;
    }
}

// Boxes, tubes and cones: FP32 decides misses, points surely inside or
// outside, and the one surface or nearest feature that FP64 has to evaluate
// (filter_pass.cuh, point_pass.cuh); the tracks that need FP64 are gathered, up to 128 per
// warp, so that 32 of one sort run together.  Points beyond the copies' reach are outside
// the solid; there the bounding sphere, with a margin that grows with the
// distance, decides misses, and the zones keep margins that grow alike.  Directions
// outside the FP32 range take the whole routine.
//
// What bounds it: the latency of the FP64 chains (FP64 unit 64 %, issue 34 %); 26 FP64
// instructions per 32 tracks of a placed cone, of which a quarter hit.  DistFromOutside of 2^20 tracks: k_shape 229 us
// (113 FP64 instructions), 66 us so.  With whole batches of 128 dealt to the warps in turn
// (1.7 for each), tracks that all need the whole routine took 15 to 30 % longer than
// k_shape (cone, 30 radii away: 252 us and 397 for the safety against 225 and 317; 29 and
// 117 so).
constexpr int kSoloWarps = 8;
constexpr int kSoloBatch = 128;
constexpr int kSoloSorts = 4;   // plane, quadric or radius, edge or corner, whole solid
struct __align__(16) SoloBatch {   // one warp's
    double p[6][kSoloBatch];
    signed char tag[kSoloBatch];
    unsigned char list[kSoloSorts][kSoloBatch];
};

// The largest coordinate of the FP32 point.  A finite point of which it is beyond the
// copies' reach (8.8 times |t| + the bounding radius) is outside the solid.
__device__ __forceinline__ float extent32(const float* p) {
    return fmaxf(fabsf(p[0]), fmaxf(fabsf(p[1]), fabsf(p[2])));
}

// Contains of boxes, tubes and cones: FP32 decides all but the points within 2 delta
// of a surface, and those cost a dozen FP64 instructions, so nothing is gathered.
__global__ void __launch_bounds__(256) k_shape_contains(const __grid_constant__ ShapeFast a, Basket b,
                                                        double* __restrict__ out, int32_t* __restrict__ face) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < b.n; i += stride) {
        const double px = b.x[i], py = b.y[i], pz = b.z[i];
        const float p[3] = {f64_to_f32_trunc(px), f64_to_f32_trunc(py), f64_to_f32_trunc(pz)};
        double v = d_nan();
        if (finite64(px) && finite64(py) && finite64(pz)) {
            int in = extent32(p) <= a.reach ? entry_holds(&a.h, p) : 0;
            if (in == 2) {
                double x[3];
                point_to_local64(a.m64, px, py, pz, x);
                in = contains64<false>(a.m64, x) ? 1 : 0;
            }
            v = in ? 1.0 : 0.0;
        }
        out[i] = v;
        if (face) face[i] = -1;
    }
}

// the whole routine (k_shape's)
template <int WHAT>
__device__ __forceinline__ double solo64(const ShapeRec64& r, double px, double py, double pz, double qx, double qy,
                                             double qz, int* f) {
    double x[3], u[3];
    to_local64(r, px, py, pz, qx, qy, qz, x, u);
    *f = -1;
    if (WHAT == GEO_Q_DIST_OUT) return dist_out64<true, false>(r, x, u, f);
    if (WHAT == GEO_Q_DIST_IN) return contains64<false>(r, x) ? dist_in64<true, false>(r, x, u, f) : 0.0;
    return safety64<false>(r, x, WHAT == GEO_Q_SAFETY_IN);
}

template <int WHAT>
__global__ void __launch_bounds__(kSoloWarps * 32, 4) k_shape_lists(const __grid_constant__ ShapeFast a, Basket b,
                                                                    double* __restrict__ out,
                                                                    int32_t* __restrict__ face) {
    constexpr bool kDist = WHAT == GEO_Q_DIST_OUT || WHAT == GEO_Q_DIST_IN;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SoloBatch& B = reinterpret_cast<SoloBatch*>(smem_raw)[warp];
    // an equal share of the basket, in whole groups of 32 tracks, for every warp
    const int64_t share = int64_t(blockIdx.x) * kSoloWarps + warp, shares = int64_t(gridDim.x) * kSoloWarps;
    const int64_t groups = (b.n + 31) >> 5, end = min((groups * (share + 1) / shares) << 5, b.n);
    for (int64_t first = (groups * share / shares) << 5; first < end; first += kSoloBatch) {
        const int per = int(min(end - first, int64_t(kSoloBatch)));
        int cnt[kSoloSorts] = {0, 0, 0, 0};
        for (int o = lane; o - lane < per; o += 32) {
            const int64_t i = first + o;
            const bool live = o < per;
            int sort = -1, tag = 0, f = -1;
            double px = 0.0, py = 0.0, pz = 0.0, qx = 1.0, qy = 0.0, qz = 0.0;
            double v = 0.0;   // where no FP64 is needed
            if (live) {
                px = b.x[i]; py = b.y[i]; pz = b.z[i];
                if (kDist) {
                    qx = b.dx[i]; qy = b.dy[i]; qz = b.dz[i];
                }
                Ray32 r;
                r.p[0] = f64_to_f32_trunc(px); r.p[1] = f64_to_f32_trunc(py); r.p[2] = f64_to_f32_trunc(pz);
                bool misses = false;
                const float extent = extent32(r.p);
                bool near = extent <= a.reach;
                if (!valid_track(px, py, pz, qx, qy, qz)) {
                    v = d_nan();
                } else {
                    if (kDist) {
                        r.d[0] = f64_to_f32_trunc(qx); r.d[1] = f64_to_f32_trunc(qy); r.d[2] = f64_to_f32_trunc(qz);
                        const float dd = fmaf(r.d[0], r.d[0], fmaf(r.d[1], r.d[1], r.d[2] * r.d[2]));
                        const bool fits = dd > a.dd_min && dd < 1e30f;
                        near = near && fits;
                        const float inv_dd = frcp(dd);
                        r.inv_dn = rsqrtf(dd) * (1.f + 4.f * kEps32f);
#pragma unroll
                        for (int k = 0; k < 3; ++k) r.e[k] = -r.d[k] * inv_dd;
                        if (WHAT == GEO_Q_DIST_OUT && !near) {
                            // far away: the line surely misses the bounding sphere, or leaves it behind
                            const float rad = fmaf(a.far, extent, a.h.brad);
                            float s0, q[3];
                            to_shifted(make_float4(a.h.t[0], a.h.t[1], a.h.t[2], 0.f), r, s0, q);
                            const float perp2 = fmaf(q[0], q[0], fmaf(q[1], q[1], q[2] * q[2]));
                            misses = fits && extent < 1e15f && (perp2 > rad * rad || fmaf(rad, r.inv_dn, s0) < 0.f);
                        }
                    }
                    if (!near) {
                        if (WHAT == GEO_Q_DIST_OUT) {
                            if (misses) v = d_inf();
                            else sort = 3;
                        } else if (WHAT == GEO_Q_SAFETY_OUT) {
                            if (extent < 1e15f) tag = entry_zone(&a.h, r.p, a.grow * extent);
                            sort = zone_sort(tag);
                        } else if (extent <= a.reach) {
                            sort = 3;   // (beyond it, from inside: 0)
                        }
                    } else if (WHAT == GEO_Q_SAFETY_OUT) {
                        tag = entry_zone(&a.h, r.p);
                        if (tag != kZoneInside) sort = zone_sort(tag);
                    } else if (WHAT == GEO_Q_DIST_OUT) {
                        Cands c;
                        cands_clear(c);
                        if (a.h.flags & kFiltBox) bound_box(&a.h, r, f_inf(), c);
                        else bound_quad(&a.h, r, f_inf(), c);
                        if (!(c.L[0] < f_inf())) {
                            v = d_inf();
                        } else {
                            tag = c.j[0] >> kTagShift;
                            if (tag != kTagNone) sort = tag == kTagOuter || tag == kTagInner ? 1 : 0;
                            else if (entry_holds(&a.h, r.p) != 1) sort = 3;   // (surely inside: 0)
                        }
                    } else {   // from inside: in the solid's own frame
                        const float4* H = hvy_words(&a.h);
                        float x[3];
                        point_to_entry(H, H[0], a.h.flags, H[3].x, r.p, x);
                        const bool surely = contains32(a.m32, x);
                        if (surely && WHAT == GEO_Q_SAFETY_IN) {
                            tag = mother_zone(a, x);
                            sort = zone_sort(tag);
                        } else if (surely) {
                            float u[3];
                            if (a.h.flags & kFiltIdentity) {
                                u[0] = r.d[0]; u[1] = r.d[1]; u[2] = r.d[2];
                            } else {
                                rotate_in(H[1], H[2], H[3].x, r.d, u);
                            }
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                r.p[k] = x[k];
                                r.d[k] = u[k];
                            }
                            tag = mother_exit32(a, r).tag;
                            sort = tag == kTagNone ? 3 : (tag == kTagOuter || tag == kTagInner ? 1 : 0);
                        } else if (contains32(a.m32u, x)) {
                            sort = 3;   // (surely outside: 0)
                        }
                    }
                }
            }
            if (live && sort < 0) {
                out[i] = v;
                if (face) face[i] = f;
            }
            if (sort >= 0) {
                B.p[0][o] = px; B.p[1][o] = py; B.p[2][o] = pz;
                if (kDist) {
                    B.p[3][o] = qx; B.p[4][o] = qy; B.p[5][o] = qz;
                }
                B.tag[o] = (signed char)tag;
                if (per <= 32 && sort < 3) sort = 0;   // (32 tracks are not worth several runs)
            }
#pragma unroll
            for (int s = 0; s < kSoloSorts; ++s) {
                const unsigned same = __ballot_sync(0xffffffffu, sort == s);
                if (sort == s) B.list[s][cnt[s] + __popc(same & ((1u << lane) - 1u))] = (unsigned char)o;
                cnt[s] += __popc(same);
            }
        }
        __syncwarp();
        for (int sort = 0, c = 0; sort < kSoloSorts;) {
            const int n = sort == 0 ? cnt[0] : (sort == 1 ? cnt[1] : (sort == 2 ? cnt[2] : cnt[3]));
            if (c >= n) {
                ++sort;
                c = 0;
                continue;
            }
            if (c + lane < n) {
                const int o = B.list[sort][c + lane], tag = B.tag[o];
                const double px = B.p[0][o], py = B.p[1][o], pz = B.p[2][o];
                const double qx = kDist ? B.p[3][o] : 0.0, qy = kDist ? B.p[4][o] : 0.0, qz = kDist ? B.p[5][o] : 0.0;
                double v;
                int f = -1;
                if (sort == 3) {
                    v = solo64<WHAT>(a.m64, px, py, pz, qx, qy, qz, &f);
                } else if (kDist) {
                    bool up = false;
                    constexpr bool kExit = WHAT == GEO_Q_DIST_IN;
                    v = surface64(a.m64, tag, kExit, px, py, pz, qx, qy, qz, &up);
                    f = tag == kTagOuter ? 6 : (tag == kTagInner ? 7 : (tag >= kTagAxis ? 2 * (tag - kTagAxis) : 4) +
                                                                           (up == kExit ? 1 : 0));
                } else {
                    v = zone64(a.m64, tag, WHAT == GEO_Q_SAFETY_IN, px, py, pz);
                }
                out[first + o] = v;
                if (face) face[first + o] = f;
            }
            __syncwarp();
            c += 32;
        }
        __syncwarp();
    }
}

template <int WHAT>
static cudaError_t launch_lists_q(const ShapeFast& a, const Basket& b, double* out, int32_t* face, cudaStream_t s,
                                  int num_sms) {
    const int smem = kSoloWarps * int(sizeof(SoloBatch));
    cudaError_t e = prep(k_shape_lists<WHAT>, smem);
    if (e != cudaSuccess) return e;
    k_shape_lists<WHAT><<<blocks_for(k_shape_lists<WHAT>, b.n, smem, num_sms), kSoloWarps * 32, smem, s>>>(a, b, out,
                                                                                                         face);
    return cudaGetLastError();
}

cudaError_t launch_shape_lists(const ShapeFast& a, int what, const Basket& b, double* out, int32_t* face,
                               cudaStream_t s, int num_sms) {
    switch (what) {
        case GEO_Q_DIST_OUT: return launch_lists_q<GEO_Q_DIST_OUT>(a, b, out, face, s, num_sms);
        case GEO_Q_DIST_IN: return launch_lists_q<GEO_Q_DIST_IN>(a, b, out, face, s, num_sms);
        case GEO_Q_SAFETY_OUT: return launch_lists_q<GEO_Q_SAFETY_OUT>(a, b, out, face, s, num_sms);
        case GEO_Q_SAFETY_IN: return launch_lists_q<GEO_Q_SAFETY_IN>(a, b, out, face, s, num_sms);
        case GEO_Q_CONTAINS:
            k_shape_contains<<<blocks_for(k_shape_contains, b.n, 0, num_sms), 256, 0, s>>>(a, b, out, face);
            return cudaGetLastError();
        default: return cudaErrorInvalidValue;
    }
}

template <int WHAT>
static cudaError_t launch_shape_q(const ShapeArg& a, const Basket& b, double* out, int32_t* face, cudaStream_t s,
                                  int num_sms) {
    k_shape<WHAT><<<blocks_for(k_shape<WHAT>, b.n, 0, num_sms), 256, 0, s>>>(a, b, out, face);
    return cudaGetLastError();
}

cudaError_t launch_shape_query(const ShapeArg& a, int what, const Basket& b, double* out, int32_t* face,
                               cudaStream_t s, int num_sms) {
    switch (what) {
        case GEO_Q_DIST_OUT: return launch_shape_q<GEO_Q_DIST_OUT>(a, b, out, face, s, num_sms);
        case GEO_Q_DIST_IN: return launch_shape_q<GEO_Q_DIST_IN>(a, b, out, face, s, num_sms);
        case GEO_Q_SAFETY_OUT: return launch_shape_q<GEO_Q_SAFETY_OUT>(a, b, out, face, s, num_sms);
        case GEO_Q_SAFETY_IN: return launch_shape_q<GEO_Q_SAFETY_IN>(a, b, out, face, s, num_sms);
        case GEO_Q_CONTAINS: return launch_shape_q<GEO_Q_CONTAINS>(a, b, out, face, s, num_sms);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace geonav
