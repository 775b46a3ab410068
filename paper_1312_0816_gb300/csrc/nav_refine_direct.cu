// nav_refine_direct.cu -- the filter step (GEO_FP32_REFINE) with one thread per
// track from the load to the store.
//
// Where the FP32 pass names the surface a track surely meets first (nearly
// every track of a volume of boxes, tubes and cones: 0.1 % are left to the
// whole routine in the toy detector), the FP64 work left is one surface
// (surface64), the same code for every kind of solid.  So there is nothing to
// sort the tracks of a tile by, and no reason to hand them from producer to
// consumer warps: each warp runs the FP32 pass of its 32 tracks, then their
// FP64 surface, and the warps of an SM overlap one another's FP32 and FP64
// phases by themselves, without barriers.
//
// What bounds it: issue slots (64 %) and the FP64 unit (62 %) together, 2900
// warp instructions and 52 FP64 instructions per 32 tracks of the toy detector
// (the pipelined kernel of refine_kernel.cuh that this one replaces there:
// 5350 and 87).  Per call, pipelined -> this: toy detector 2^20 tracks 218 ->
// 140 us, 65536 tracks 34.8 -> 23.3 us; four boxes 122 -> 43.6 us and 15.0 ->
// 8.7 us; 512 rotated solids without the grid 982 -> 649 us and 121 -> 83 us.
// Four blocks of 256 threads per SM (64 registers): 143.6 us for the toy
// detector's 2^20 tracks through the binding; three blocks 148, two 160, eight of 128
// threads 146, sixteen of 64 threads 161.  Volumes with tube segments or polycones keep the pipelined
// kernel: their tracks need whole solids of differing kinds, which its bins
// keep apart (four polycones, 300007 tracks: 276 us here, 147 us there).
#include <cuda_runtime.h>

#include "geo_internal.h"
#include "launch.cuh"
#include "nav_common.cuh"
#include "nav_refine.cuh"
#include "stage.cuh"

namespace geonav {

constexpr int kDirect = 256;         // threads per block
constexpr int kDirectBlocks = 4;     // resident blocks per SM

template <int SMEM>
__global__ void __launch_bounds__(kDirect, kDirectBlocks)
    k_dist_direct(const __grid_constant__ VolView v, Basket b, double* __restrict__ step, int32_t* __restrict__ hit,
                  double* __restrict__ bpoint, int32_t* __restrict__ nref) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bar;
    __shared__ ShapeRec64 m64;        // the mother's record beside the daughters'
    __shared__ double pd[6][kDirect];   // each thread's track, so that it does not live in registers
    FiltTab f = {v.fsph, v.fhvy, v.nq1, v.nq, v.nf};
    const ShapeRec64* tab64 = v.d64;
    const int t = threadIdx.x;
    if (t < int(sizeof(ShapeRec64) / sizeof(double)))
        reinterpret_cast<double*>(&m64)[t] = reinterpret_cast<const double*>(&v.m64)[t];
    if (SMEM) {
        const uint32_t bf = uint32_t(v.nf) * uint32_t(sizeof(FiltSph) + sizeof(FiltHvy));
        if (!stage_tables(smem_raw, v.fsph, bf, smem_raw + bf, v.d64,
                          SMEM == 2 ? uint32_t(v.nd) * uint32_t(sizeof(ShapeRec64)) : 0, &bar, v.status))
            return;
        f.sph = reinterpret_cast<const FiltSph*>(smem_raw);
        f.hvy = reinterpret_cast<const FiltHvy*>(smem_raw + size_t(v.nf) * sizeof(FiltSph));
        if (SMEM == 2) tab64 = reinterpret_cast<const ShapeRec64*>(smem_raw + bf);
    }
    __syncthreads();
    const int64_t stride = int64_t(gridDim.x) * kDirect;
    for (int64_t i = int64_t(blockIdx.x) * kDirect + t; i < b.n; i += stride) {
        RefineState rs;
        double best = 0.0;
        int h = -2, nev = 0;
        {
            const double px = b.x[i], py = b.y[i], pz = b.z[i];
            const double qx = b.dx[i], qy = b.dy[i], qz = b.dz[i];
            pd[0][t] = px; pd[1][t] = py; pd[2][t] = pz;
            pd[3][t] = qx; pd[4][t] = qy; pd[5][t] = qz;
            asm volatile("" ::: "memory");   // read again below
            refine_pass1<kTravAll, false>(v, f, GridTab{}, tab64, px, py, pz, qx, qy, qz, [&](int c) { return pd[c][t]; }, rs, best, h,
                                     nev);
        }
        const double px = pd[0][t], py = pd[1][t], pz = pd[2][t], qx = pd[3][t], qy = pd[4][t], qz = pd[5][t];
        finish_direct(v, tab64, m64, rs, px, py, pz, qx, qy, qz, best, h, nev);
        store_result(i, b.n, best, h, px, py, pz, qx, qy, qz, step, hit, bpoint);
        if (nref) nref[i] = nev;
    }
}

template <int SMEM>
static cudaError_t launch_direct(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                                 int32_t* nref, cudaStream_t s, int num_sms) {
    const int smem = (SMEM ? v.nf * int(sizeof(FiltSph) + sizeof(FiltHvy)) : 0) +
                     (SMEM == 2 ? v.nd * int(sizeof(ShapeRec64)) : 0);
    auto kernel = k_dist_direct<SMEM>;
    cudaError_t e = prep(kernel, smem);
    if (e != cudaSuccess) return e;
    kernel<<<blocks_for(kernel, b.n, smem, num_sms, kDirect), kDirect, smem, s>>>(v, b, step, hit, bpoint, nref);
    return cudaGetLastError();
}

cudaError_t launch_dist_direct(const VolView& v, const Basket& b, double* step, int32_t* hit, double* bpoint,
                               int32_t* nref, cudaStream_t s, int num_sms) {
    if (v.voxelized) return launch_dist_grid(v, b, step, hit, bpoint, nref, s, num_sms);
    if (v.smem_refine == 2) return launch_direct<2>(v, b, step, hit, bpoint, nref, s, num_sms);
    if (v.smem_refine == 1) return launch_direct<1>(v, b, step, hit, bpoint, nref, s, num_sms);
    return launch_direct<0>(v, b, step, hit, bpoint, nref, s, num_sms);
}

}  // namespace geonav
