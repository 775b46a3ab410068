// world_direct.cu -- the filtered step of a geometry tree whose volumes hold
// boxes, tubes and cones alone: one thread per track from the load to the
// store (see nav_refine_direct.cu).  The tracks come grouped by logical volume
// (world.cu), so the lanes of a warp mostly read one volume's tables; a warp
// that spans two volumes takes them one after the other.
//
// After its FP32 pass a track's FP64 work is one surface of its first solid,
// the re-entry of the daughter it has just left where FP32 cannot rule that
// out (a convex solid is never entered again), and the relocation.
//
// What bounds it: the FP64 unit (49 %: 79 FP64 instructions per 32 tracks, of
// which the transform into a rotated node 21) and the latency of the grouped
// order's gathers.  Toy world, 2^20 tracks after two steps, the whole call:
// 567 us with k_world_step_binned and the scatter's global atomics, 281 us so
// (three blocks per SM 298, two 313); the step kernel alone 454 -> 255 us.
#include <cuda_runtime.h>

#include "launch.cuh"
#include "world.cuh"

namespace geonav {

constexpr int kWorldThreads = 256;
constexpr int kWorldBlocks = 4;   // resident blocks per SM (64 registers)

// FP32 pass (world_pass1's answers and bounds); re: what FP32 knows of the
// re-entry into `skip`, reL a lower bound of it.
template <class Src>
__device__ __forceinline__ void world_pass_lists(const VolView& v, const double* x, const double* u, Src src, int skip,
                                                 bool entered, RefineState& st, double& best, int& h, int& re,
                                                 float& reL) {
    st.status = 1;
    cands_clear(st.c);
    st.Lm = 0.f;
    re = kReentryNone;
    reL = 0.f;
    if (!valid_track(x[0], x[1], x[2], u[0], u[1], u[2])) {
        best = d_nan();
        h = -2;
        return;
    }
    Ray32 r;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r.p[k] = f64_to_f32_trunc(x[k]);
        r.d[k] = f64_to_f32_trunc(u[k]);
    }
    const float dd = fmaf(r.d[0], r.d[0], fmaf(r.d[1], r.d[1], r.d[2] * r.d[2]));
    if (!(dd > v.dd_min && dd < 1e30f)) {
        const double xx[3] = {src(0), src(1), src(2)}, uu[3] = {src(3), src(4), src(5)};
        world_nav64(v, xx, uu, skip, entered, best, h);
        return;
    }
    const float inv_dd = __frcp_rn(dd);
    r.inv_dn = rsqrtf(dd) * (1.f + 4.f * kEps32f);
#pragma unroll
    for (int k = 0; k < 3; ++k) r.e[k] = -r.d[k] * inv_dd;
    const MotherExit m = mother_exit32<true>(v, r, entered);
    if (!(m.in || entered || contains64_cold<false>(v.m64, src(0), src(1), src(2)))) {
        best = 0.0;
        h = -2;
        return;
    }
    st.Lm = m.in ? fmaxf(lower_bound(m.lo, v.m32.delta, r.inv_dn), 0.f) : 0.f;
    const float Um = m.hi + 16.f * kEps32f * m.hi + v.m32u.delta * r.inv_dn;
    const int ke = skip >= 0 ? v.fhvy[skip].entry : -1;
    const FiltTab f = {v.fsph, v.fhvy, v.nq1, v.nq, v.nf};
    filter_daughters<true>(f, r, Um, st.c, ke);
    if (skip >= 0) re = reentry32(v.fhvy + ke, r, reL);
    st.tag = first_task(st) < 0 ? m.tag : st.c.j[0] >> kTagShift;
#pragma unroll
    for (int k = 0; k < kCand; ++k) st.c.j[k] &= kIdMask;
    st.status = 0;
}

static __device__ __noinline__ double reentry64_cold(const ShapeRec64& r, double x0, double x1, double x2, double u0,
                                                     double u1, double u2) {
    double xl[3], ul[3];
    to_local64(r, x0, x1, x2, u0, u1, u2, xl, ul);
    return reentry64(r, xl, ul);
}

__global__ void __launch_bounds__(kWorldThreads, kWorldBlocks)
    k_world_step_direct(WorldView w, Basket b, const int32_t* __restrict__ perm, const int32_t* __restrict__ node_in,
                        const int32_t* __restrict__ flag_in, double* __restrict__ step, int32_t* __restrict__ node_out,
                        int32_t* __restrict__ flag_out) {
    __shared__ double pd[6][kWorldThreads];   // each thread's track in its node's frame
    const int tid = threadIdx.x;
    const int64_t stride = int64_t(gridDim.x) * kWorldThreads;
    for (int64_t t = int64_t(blockIdx.x) * kWorldThreads + tid; t < b.n; t += stride) {
        const int64_t i = perm[t];
        const int node = node_in[i];
        const int flag = flag_in ? flag_in[i] : -1;
        double best = d_nan();
        int nout = -2, fout = -1;
        if (node >= 0 && node < w.nnodes) {
            const VolView& v = w.vols[w.lv[node]];
            const int skip = flag >= 0 && flag < v.nd ? flag : -1;
            RefineState st;
            int h = -2, re;
            float reL;
            {
                double x[3], u[3];
                world_to_node(w.xf + 12 * size_t(node), b.x[i], b.y[i], b.z[i], b.dx[i], b.dy[i], b.dz[i], x, u);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    pd[k][tid] = x[k];
                    pd[3 + k][tid] = u[k];
                }
                asm volatile("" ::: "memory");   // read again below
                world_pass_lists(v, x, u, [&](int c) { return pd[c][tid]; }, skip, flag == -2, st, best, h, re, reL);
            }
            const double x[3] = {pd[0][tid], pd[1][tid], pd[2][tid]}, u[3] = {pd[3][tid], pd[4][tid], pd[5][tid]};
            if (st.status == 0) {
                const int task = first_task(st);
                double s1;
                if (st.tag != kTagNone)
                    s1 = surface64(task < 0 ? v.m64 : v.d64[task], st.tag, task < 0, x[0], x[1], x[2], u[0], u[1], u[2]);
                else s1 = eval64_cold(v, v.d64, task, x[0], x[1], x[2], u[0], u[1], u[2]);
                int nev = 0;
                if (!refine_fast(st, s1, best, h))
                    refine_rest<false>(v, v.d64, st, s1, x[0], x[1], x[2], u[0], u[1], u[2], best, h, nev);
                if (nev >= 1000) {   // the candidate list overflowed: the loop over every daughter
                    world_nav64(v, x, u, skip, flag == -2, best, h);
                } else if (skip >= 0 && re != kReentryNone && reL <= f64_to_f32_up(best)) {
                    const ShapeRec64& r = v.d64[skip];
                    const double s = re != kTagNone ? surface64(r, re, false, x[0], x[1], x[2], u[0], u[1], u[2])
                                                    : reentry64_cold(r, x[0], x[1], x[2], u[0], u[1], u[2]);
                    if (LT(s, best) || (BITS(s) == BITS(best) && h >= 0 && skip < h)) {
                        best = s;
                        h = skip;
                    }
                }
            }
            if (h >= -1) {
                double bp[3] = {FMA(best, u[0], x[0]), FMA(best, u[1], x[1]), FMA(best, u[2], x[2])};
                world_relocate(w, node, h, bp, nout, fout);
            }
        }
        step[i] = best;
        node_out[i] = nout;
        if (flag_out) flag_out[i] = fout;
    }
}

cudaError_t launch_world_step_direct(const WorldView& w, const Basket& b, const int32_t* perm, const int32_t* node_in,
                                     const int32_t* flag_in, double* step, int32_t* node_out, int32_t* flag_out,
                                     cudaStream_t s, int num_sms) {
    k_world_step_direct<<<blocks_for(k_world_step_direct, b.n, 0, num_sms, kWorldThreads), kWorldThreads, 0, s>>>(
        w, b, perm, node_in, flag_in, step, node_out, flag_out);
    return cudaGetLastError();
}

}  // namespace geonav
